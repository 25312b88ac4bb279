// npm_tc.cu -- tensor-core path on sm_103a: the training kernel, the
// arrangement of the weights for the MMAs, the model's tensor-core state and
// the dispatch of the forward kernels (npm_tc_forward.cuh, npm_tc_tiny.cu).
//
// The training kernel runs groups of 256 threads over 128-sample tiles, two
// threads per sample: two groups a CTA that share the weights, or one group and
// up to three CTAs an SM. Activations and gradients are BF16 operand tiles in
// shared memory (planes of 8 columns), one elected thread of a group issues
// tcgen05.mma kind::f16 with FP32 accumulation in tensor memory and commits
// to an mbarrier, and the threads read their accumulator lanes with
// tcgen05.ld. Weights arrive once per CTA by a bulk asynchronous copy. Every
// wait on an mbarrier is bounded: on timeout the kernel records
// NPM_ERR_TIMEOUT in the status word, releases its tensor memory and returns.
#include <cuda_bf16.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "npm_handle.h"
#include "npm_kernels.h"
#include "npm_tc.cuh"

namespace npm {

using namespace tc;

namespace {

// Place of a value in an operand tile stored in planes (kPlane): a tile and the
// residual tile behind it are one operand of twice the columns.
__device__ __forceinline__ uint32_t plane_off(int row, int col) {
    return (uint32_t)(col >> 3) * kPlane + (uint32_t)row * 16u + (uint32_t)(col & 7) * 2u;
}

// --------------------------------------------------------------- encode

// The inputs of one training sample from the FP32 table: row `row` of the
// tile at sA, residuals lo bytes further. F2: 2 features per level
// (compile-time). Levels [lbeg, lend) are encoded; tail: also the
// product-mode inputs and the zero padding to kp columns.
template <bool F2>
__device__ __forceinline__ void tc_encode(const TcCfg& tc, const float* __restrict__ grid32, int64_t j, bool valid,
                                          int64_t ld, const float* __restrict__ pos, const float* __restrict__ aux,
                                          uint8_t* sA, int row, uint32_t lo, int lbeg, int lend, bool tail) {
    const DevCfg& cfg = tc.base;
    float x = 0.0f, y = 0.0f, z = 0.0f;
    if (valid) {
        x = pos[j];
        y = pos[ld + j];
        z = pos[2 * ld + j];
    }
    const int F = F2 ? 2 : cfg.feat;
    for (int l = lbeg; l < lend; ++l) {
        const Cell cl = make_cell(x, y, z, cfg.level_res[l]);
        if (F2) {
            Level2<float> v;
            v.load_table(cfg, grid32, l, cl);
            const float2 a = v.blend(cl);
            store_pair(sA, plane_off(row, 2 * l), a.x, a.y, lo);
            continue;
        }
        const float* gl = grid32 + (size_t)cfg.level_off[l] * F;
        uint32_t idx[8];
        corner_idx8(cfg, l, cl, idx);
        if (F == 4 || F == 8) {
            // One vector load per corner and group of 4 features.
            for (int h = 0; h < (F >> 2); ++h) {
                float4 raw[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) raw[c] = load_raw4(gl, idx[c], F, h);
                float ws[8];
                corner_w8(cl, ws);
                float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    acc.x = fmaf(ws[c], raw[c].x, acc.x);
                    acc.y = fmaf(ws[c], raw[c].y, acc.y);
                    acc.z = fmaf(ws[c], raw[c].z, acc.z);
                    acc.w = fmaf(ws[c], raw[c].w, acc.w);
                }
                const int k = l * F + 4 * h;
                store_pair(sA, plane_off(row, k), acc.x, acc.y, lo);
                store_pair(sA, plane_off(row, k + 2), acc.z, acc.w, lo);
            }
        } else {  // F = 1
            float ws[8], s = 0.0f;
            corner_w8(cl, ws);
#pragma unroll
            for (int c = 0; c < 8; ++c) s = fmaf(ws[c], __ldg(gl + idx[c]), s);
            store_one(sA, plane_off(row, l), s, lo);
        }
    }
    if (!tail) return;
    int k = cfg.grid_feats;
    if (cfg.mode == NPM_PRODUCT) {
        float e[21];
        float wo[3] = {0.0f, 0.0f, 1.0f}, nn[3] = {0.0f, 0.0f, 1.0f}, r = 0.0f;
        if (valid) {
            wo[0] = aux[j];
            wo[1] = aux[ld + j];
            wo[2] = aux[2 * ld + j];
            nn[0] = aux[3 * ld + j];
            nn[1] = aux[4 * ld + j];
            nn[2] = aux[5 * ld + j];
            r = aux[6 * ld + j];
        }
        sh_band4(wo[0], wo[1], wo[2], e);
        sh_band2(nn[0], nn[1], nn[2], e + 16);
        e[20] = r;
#pragma unroll
        for (int i = 0; i < 21; ++i) store_one(sA, plane_off(row, k + i), e[i], lo);
        k += 21;
    }
    for (; k < tc.layer[0].Kp; ++k) store_one(sA, plane_off(row, k), 0.0f, lo);
}

// Master FP32 weights (packed [out][in] per layer) -> 16-bit operand parts in
// the UMMA K-major layout, zero padded to Np x Kp per layer; with wfwd also
// the CUDA-core kernels' padded copy. blockIdx.y: layer (one pass of load latency for all layers
// instead of one each).
__global__ void k_tc_weights(const __grid_constant__ TcCfg tc, const float* mlp, uint8_t* __restrict__ blob,
                             float* __restrict__ wfwd, UpdateEnd end) {
    grid_dep_wait();
    const int l = blockIdx.y;
    if (l == 0 && blockIdx.x == 0 && threadIdx.x == 0) end_update(end);
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    if (wfwd) arrange_layer(tc.base, l, mlp, wfwd, tid, nt);
    const TcLayer& ly = tc.layer[l];
    for (int m = 0; m < l; ++m) mlp += tc.layer[m].K * tc.layer[m].N;
    // Whole rows (outputs) at a time, a thread per weight.
    const int rows = (int)blockDim.x / ly.Kp, r = (int)threadIdx.x / ly.Kp, k = (int)threadIdx.x % ly.Kp;
    bool nan = false;
    for (int nn = blockIdx.x * rows + r; r < rows && nn < ly.Np; nn += gridDim.x * rows) {
        const float v = (nn < ly.N && k < ly.K) ? mlp[nn * ly.K + k] : 0.0f;
        nan = nan || isnan(v);
        uint8_t* at = blob + ly.w_off + tile_off(nn, k, ly.Kp);
        if (tc.f16) {
            // FP16 high part and FP16 residual (the weights to ~22 bits)
            const __half hh = __float2half_rn(v);
            *reinterpret_cast<__half*>(at) = hh;
            *reinterpret_cast<__half*>(at + tc.w_bytes) = __float2half_rn(v - __half2float(hh));
            continue;
        }
        // BF16 parts, each rounded to nearest from what the ones before
        // leave (three hold all 24 bits).
        float rest = v;
        for (int p = 0; p < tc.wparts; ++p) {
            __nv_bfloat16 b = __float2bfloat16_rn(rest);
            if (tc.wparts == 3 && p == 0 && __hisinf(b)) b = __float2bfloat16_rz(copysignf(3.38e38f, rest));
            *reinterpret_cast<__nv_bfloat16*>(at + p * tc.w_bytes) = b;
            rest -= __bfloat162float(b);
        }
    }
    // FP32 arithmetic: a NaN weight makes its output NaN for every query, which
    // a hidden layer's ReLU takes for zero (three_bf16). Rare: the rows of this
    // block that hold one are cleared once all are written.
    if (tc.wparts == 3 && l + 1 < tc.base.n_layers && __syncthreads_or(nan))
        for (int nn = blockIdx.x * rows + r; r < rows && nn < ly.N; nn += gridDim.x * rows)
            if (k < ly.K && isnan(mlp[nn * ly.K + k]))
                for (int i = 0; i < 3 * ly.Kp; ++i)
                    *reinterpret_cast<uint16_t*>(blob + ly.w_off + tile_off(nn, i / 3, ly.Kp) + (i % 3) * tc.w_bytes) = 0;
}

// ------------------------------------------------------- corner blocks

// Entries of a chunk of corner blocks (kept up to date as a whole).
constexpr int kBlkChunk = 1024;
// Queries from which a batch uses them. Without and with blocks that are up to
// date (GB300, us; 2^18 and 2^20 queries): paper-shaped hash grid in FP32 110
// and 97, 398 and 343, in FP16 86 and 70, 288 and 229; eight dense levels of
// four features in FP32 83 and 73, in FP16 55 and 43, 204 and 140. At 2^17 they
// give 0 to 6 us. The first batch after an update also pays for bringing them
// up to date, 11 to 13 us on the hash grid and 16 on the dense levels, as does
// every batch of an FP32 model whose address was handed out: with an update
// before each batch they repay that from a few hundred thousand queries on.
constexpr int64_t kBlkMinQueries = 1 << 18;

// Rewrites the chunks of corner blocks whose parameters have changed since
// (built[chunk] != *version), or all where the table may have changed unseen
// (shared not NULL and *shared not zero). Each chunk's mark is set by the
// thread block that wrote all of it, so that launches on several streams may
// overlap: they write the same bytes, and a query sees its own stream's
// launch complete. Bound by its writes: 33 MB for 1.02 M entries.
template <typename GT, int F>
__global__ void __launch_bounds__(256) k_corner_blocks(const __grid_constant__ TcCfg tc, const GT* __restrict__ table,
                                                       uint4* __restrict__ blk, uint32_t total,
                                                       int* __restrict__ built, const int* __restrict__ version,
                                                       const int* __restrict__ shared) {
    constexpr int C = blk_corners(F, sizeof(GT)), V = 8 / C;  // corners, 32-bit values a corner
    __shared__ int now, stale;
    grid_dep_launch();
    if (threadIdx.x == 0) {
        now = *version;
        stale = built[blockIdx.x] != now || (shared && *shared);
    }
    __syncthreads();
    if (!stale) return;
    const DevCfg& cfg = tc.base;
    const uint32_t* t32 = reinterpret_cast<const uint32_t*>(table);
    for (uint32_t e = blockIdx.x * kBlkChunk + threadIdx.x; e < min(total, (blockIdx.x + 1) * kBlkChunk);
         e += blockDim.x) {
        int l = -1;  // the last level with blocks that starts at or before e
        for (int m = 0; m < cfg.n_levels; ++m)
            if (((tc.blk_mask >> m) & 1u) && tc.blk_off[m] <= e) l = m;
        const uint32_t D = (uint32_t)cfg.level_res[l], i = e - tc.blk_off[l], last = D * D * D - 1u;
        uint32_t r[8];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            // (entries past the level's end belong to no cell)
            const uint32_t at = cfg.level_off[l] + min(i + (c & 1) + ((c & 2) ? D : 0u) + ((c & 4) ? D * D : 0u), last);
#pragma unroll
            for (int q = 0; q < V; ++q) r[c * V + q] = t32[(size_t)at * V + q];
        }
        blk[2 * (size_t)e] = make_uint4(r[0], r[1], r[2], r[3]);
        blk[2 * (size_t)e + 1] = make_uint4(r[4], r[5], r[6], r[7]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) built[blockIdx.x] = now;
}

// ----------------------------------------------------------- training

// Training layout. A CTA holds G tile groups of 256 threads that share the
// weights and the weight-gradient accumulators; each group walks its own
// 128-sample tiles. A group's shared memory is one slot per layer, slot l with
// the BF16 high parts of layer l's input (kPlane layout), and a last slot L:
//   forward  : slot L holds the residuals of the current layer's input;
//   loss     : the loss gradient, high parts and residuals, goes to slot L;
//   backward : the gradient of layer l's input replaces that input in slot l,
//              its residuals follow in slot l + 1, whose contents (the
//              gradient of layer l's output) the finished MMAs have read.
// So a gradient and its residuals are always adjacent, and where both fit 128
// rows one MMA per K step forms D_hi^T H and D_lo^T H in lanes o and Np + o of
// the layer's accumulator. (The MMA reads 128 rows: what lies behind the
// tiles, at most 32 KB from a slot's start, ends in lanes never read.)
// Tensor memory: every layer's weight gradient (Kp_l columns, all tiles of the
// CTA), then per group an accumulator and the parked encoder gradient.
struct TcTrain {
    uint32_t slot[NPM_MAX_LAYERS + 1];  // byte offsets within a group's tiles
    uint32_t dw_col[NPM_MAX_LAYERS];
    uint32_t idesc_dw[NPM_MAX_LAYERS];  // A MN-major, B MN-major, N = Kp_l
    uint32_t idesc_dx[NPM_MAX_LAYERS];  // A K-major,  B MN-major, N = Kp_l
    uint32_t g_bytes;                   // a group's tiles
    uint32_t x_off, w_off, bar_off, smem;
    uint32_t acc_col, acc_cols, park_col, tmem_cols;
    int64_t woff[NPM_MAX_LAYERS];       // packed offset of W_l in the MLP region
    int groups;
    int park;                           // encoder gradients wait in tensor memory (2-feature grids)
};

// Training runs two threads per sample row: thread t of a group serves row
// t & 127 and half t >> 7 of the row's work (grid levels, epilogue column
// chunks, lobes). Warps w and w + 4 read the same TMEM lane quarter.
constexpr int kTrainThreads = 2 * kTile;

// Named barrier of training group g (id 0 is the CTA's), and its form that
// also ORs a predicate.
__device__ __forceinline__ void train_sync(int g) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kTrainThreads) : "memory");
}
__device__ __forceinline__ bool train_sync_or(int g, bool p) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred q, o;\n\t"
        "setp.ne.u32 q, %3, 0;\n\t"
        "bar.red.or.pred o, %1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, o;\n\t}\n"
        : "=r"(r)
        : "r"(1 + g), "r"(kTrainThreads), "r"((uint32_t)p)
        : "memory");
    return r != 0;
}

// Turns at the shared weight-gradient accumulators: MMAs of two threads are
// not ordered by themselves, so a group's thread takes the turn, waits for the
// completion of the batch before (its commit's phase of `bar`), issues and
// commits its own, and passes the turn on without waiting for it.
struct DwTurn {
    uint32_t taken;    // 0 or 1
    uint32_t batches;  // batches issued so far
};
__device__ __forceinline__ bool take_turn(DwTurn* turn, uint32_t bar) {
    const long long t0 = clock64();
    while (atomicCAS(&turn->taken, 0u, 1u) != 0u) {
        if (clock64() - t0 > (1ll << 32)) return false;
        __nanosleep(20);
    }
    __threadfence_block();
    const uint32_t b = *reinterpret_cast<volatile uint32_t*>(&turn->batches);
    if (b > 0 && !mbar_wait_bounded(bar, (b - 1) & 1u)) {
        atomicExch(&turn->taken, 0u);
        return false;
    }
    return true;
}
__device__ __forceinline__ void pass_turn(DwTurn* turn) {
    *reinterpret_cast<volatile uint32_t*>(&turn->batches) += 1u;
    __threadfence_block();
    atomicExch(&turn->taken, 0u);
}

// Half h of the lobes of one sample, lobes i = h KMAX/2 + q. Pass 1 forms
// each lobe's terms and the half's partial log-sum-exps of the softmax
// logits (m1, s1) and of the unnormalised log lobe values
// a'_i = raw_i + log c(kappa_i) + kappa_i (mu_i.w - 1) (m2, s2); the caller
// combines both halves' partials (log V = LSE(a') - LSE(raw)).
template <int KMAX>
struct GradHalf {
    static constexpr int KH = KMAX / 2;
    float r0[KH], ap[KH], kap[KH], md[KH], wdt[KH], wdp[KH], sk[KH], st[KH], sp[KH];
    bool act[KH];

    __device__ __forceinline__ float4 pass1(const DevCfg& cfg, int h, const float (&raw)[4 * KH], const float w[3]) {
        float m1 = -INFINITY, m2 = -INFINITY;
#pragma unroll
        for (int q = 0; q < KH; ++q) {
            act[q] = h * KH + q < cfg.K;
            r0[q] = raw[4 * q];
            const float rk = raw[4 * q + 1];
            if (cfg.kappa_act == NPM_EXP) {
                kap[q] = __expf(rk);
                sk[q] = kap[q];
            } else {
                // softplus and its derivative, the logistic, from one e^{-|rk|}
                const float e = __expf(-fabsf(rk));
                const float r1 = __fdividef(1.0f, 1.0f + e);
                kap[q] = fmaxf(rk, 0.0f) + __logf(1.0f + e);
                sk[q] = rk >= 0.0f ? r1 : e * r1;
            }
            st[q] = logistic_fast(raw[4 * q + 2]);
            sp[q] = logistic_fast(raw[4 * q + 3]);
            // theta = pi st, phi = pi + pi (2 sp - 1): sine/cosine on [-pi, pi]
            float sth, cth, sph, cph;
            __sincosf(kPi * st[q] - 0.5f * kPi, &cth, &sth);
            cth = -cth;
            __sincosf(kPi * (2.0f * sp[q] - 1.0f), &sph, &cph);
            sph = -sph;
            cph = -cph;
            md[q] = sth * cph * w[0] + sth * sph * w[1] + cth * w[2];
            wdt[q] = cth * cph * w[0] + cth * sph * w[1] - sth * w[2];
            wdp[q] = -sth * sph * w[0] + sth * cph * w[1];
            ap[q] = r0[q] + __logf(vmf_scaled_norm_fast(kap[q])) + kap[q] * (md[q] - 1.0f);
            if (act[q]) {
                m1 = fmaxf(m1, r0[q]);
                m2 = fmaxf(m2, ap[q]);
            }
        }
        float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
        for (int q = 0; q < KH; ++q)
            if (act[q]) {
                s1 += __expf(r0[q] - m1);
                s2 += __expf(ap[q] - m2);
            }
        return make_float4(m1, s1, m2, s2);
    }

    // s d log V / d raw of this half's lobes (zero for lobes beyond K).
    __device__ __forceinline__ void pass2(float lse, float lsa, float s, float (&d)[4 * KH]) const {
#pragma unroll
        for (int q = 0; q < KH; ++q) {
            if (act[q]) {
                const float r = __expf(ap[q] - lsa);   // posterior of lobe q
                const float lam = __expf(r0[q] - lse); // its mixture weight
                const float sr = s * r;
                d[4 * q + 0] = s * (r - lam);
                d[4 * q + 1] = sr * (inv_minus_coth(kap[q]) + md[q]) * sk[q];
                d[4 * q + 2] = sr * kap[q] * wdt[q] * kPi * st[q] * (1.0f - st[q]);
                d[4 * q + 3] = sr * kap[q] * wdp[q] * 2.0f * kPi * sp[q] * (1.0f - sp[q]);
            } else {
                d[4 * q + 0] = d[4 * q + 1] = d[4 * q + 2] = d[4 * q + 3] = 0.0f;
            }
        }
    }
};

// log(e^{m_a} s_a + e^{m_b} s_b) for partial sums that may be empty (s = 0).
__device__ __forceinline__ float lse_combine(float ma, float sa, float mb, float sb) {
    const float m = fmaxf(ma, mb);
    float t = 0.0f;
    if (sa > 0.0f) t += sa * __expf(ma - m);
    if (sb > 0.0f) t += sb * __expf(mb - m);
    return m + __logf(t);
}

// NC (a multiple of 8) values as BF16 at row t, columns c0 .. c0+NC of a tile
// in planes, with their residuals lo_off bytes on.
template <int NC>
__device__ __forceinline__ void store_cols(uint8_t* base, int t, int c0, const float* v, uint32_t lo_off) {
#pragma unroll
    for (int c = 0; c < NC; c += 8) {
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162 hb = __floats2bfloat162_rn(v[c + 2 * i], v[c + 2 * i + 1]);
            hw[i] = *reinterpret_cast<uint32_t*>(&hb);
            const float2 hf = __bfloat1622float2(hb);
            lw[i] = pack_bf16(v[c + 2 * i] - hf.x, v[c + 2 * i + 1] - hf.y);
        }
        const uint32_t off = plane_off(t, c0 + c);
        *reinterpret_cast<uint4*>(base + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(base + lo_off + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
    }
}

// Encoder-gradient scatter (Eq. 11 transposed) of levels lbeg .. lbeg+NLV
// with FF features per level; dg holds their 16 columns.
template <int FF, int NLV>
__device__ __forceinline__ void scatter_levels(const DevCfg& cfg, float* __restrict__ grad, float x, float y,
                                               float z, int lbeg, const float (&dg)[16]) {
#pragma unroll
    for (int q = 0; q < NLV; ++q) {
        const int l = lbeg + q;
        if (l < cfg.n_levels) {
            const Cell cl = make_cell(x, y, z, cfg.level_res[l]);
            float* gl = grad + (size_t)cfg.level_off[l] * FF;
            uint32_t idx[8];
            float ws[8];
            corners8(cfg, l, cl, idx, ws);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float wc = ws[c];
                float* e = gl + (size_t)idx[c] * FF;
                if constexpr (FF == 1) {
                    red_add(e, wc * dg[q]);
                } else if constexpr (FF == 2) {
                    if (c & 1) continue;  // corners c, c + 1 (along x) together
                    scatter_pair2(gl, cfg.level_off[l] + cfg.grid_shift, idx[c], idx[c + 1], ws[c], ws[c + 1], dg[2 * q],
                                  dg[2 * q + 1]);
                } else {
#pragma unroll
                    for (int f = 0; f < FF; f += 4)
                        red_add(e + f, wc * dg[FF * q + f], wc * dg[FF * q + f + 1], wc * dg[FF * q + f + 2],
                                wc * dg[FF * q + f + 3]);
                }
            }
        }
    }
}

// Grid features of a training batch for 2-feature grids (Sec. 5.1, Eq. 11):
// enc[l][j] = sum_corners w_c V_l[corner] (two values) from the FP32 master
// table. One thread per sample and kEncLevels levels (blockIdx.y: level
// group), so that a warp reads and writes one level at a time; a
// full-occupancy kernel without shared memory keeps the whole L1 and many
// warps for these random L2 reads, which the training kernel (one CTA per SM
// holding most of the shared memory) cannot. Bound by the L1's one request
// per lane and cycle. 2^19 samples of the 16-level grid (GB300): 138 us with
// 2 levels a thread, 139 with 1, 150 with 4; 174 with a warp's lanes spread
// over the levels of four samples; whole 32-byte sectors per pair (5 instead
// of 6 requests a level, more registers) 154.
constexpr int kEncLevels = 2;

__global__ void __launch_bounds__(256) k_train_encode(const __grid_constant__ DevCfg cfg,
                                                      const float* __restrict__ grid32, int64_t n,
                                                      int64_t ld, const float* __restrict__ pos,
                                                      float2* __restrict__ enc) {
    const int l0 = (int)blockIdx.y * kEncLevels;
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= n) return;
    const float x = pos[j], y = pos[ld + j], z = pos[2 * ld + j];
    Cell cs[kEncLevels];
    Level2<float> v[kEncLevels];
#pragma unroll
    for (int r = 0; r < kEncLevels; ++r)
        if (l0 + r < cfg.n_levels) {
            cs[r] = make_cell(x, y, z, cfg.level_res[l0 + r]);
            v[r].load_table(cfg, grid32, l0 + r, cs[r]);
        }
#pragma unroll
    for (int r = 0; r < kEncLevels; ++r)
        if (l0 + r < cfg.n_levels) enc[(int64_t)(l0 + r) * n + j] = v[r].blend(cs[r]);
}

// CTAs per SM of the one-group instances: three for the small four-lobe one
// (single-level grids; 80 registers without spills, 53 KB a CTA), whose tile
// chain of MMA round trips is latency-bound and overlapped by the other CTAs.
// (Four CTAs at 64 registers measured slower.) The multi-level networks
// overlap two tiles in one CTA instead: two groups share the weights.
// Measured against one tile of 256 threads a CTA (GB300): product-mode
// network, 2^19 samples, kernel 610 -> 451 us, with vector reductions in the
// place of atomics on vectors (which return their result; 972 us with them)
// and the flush of the weight gradients below (383 us with elect_one and the
// deferred scatter's turns as well); small network, 2^18 samples, 100 -> 82 us
// (165 us with one scalar atomic per weight and share), now 67.
__host__ __device__ constexpr int train_ctas_per_sm(int kmax, bool f2, int g) {
    return g == 1 && kmax == 4 && !f2 ? 3 : 1;
}

template <int KMAX, bool F2, int G>
__global__ void __launch_bounds__(kTrainThreads* G, train_ctas_per_sm(KMAX, F2, G)) k_train_tc(
    const __grid_constant__ TcCfg tc, const __grid_constant__ TcTrain tt, const float* __restrict__ grid32,
    const uint8_t* __restrict__ wblob, int64_t n, int64_t ld, const float* __restrict__ pos,
    const float* __restrict__ aux, const float* __restrict__ dir, const float* __restrict__ rad,
    const float* __restrict__ spdf, const float* __restrict__ dlogv, float inv_n, float* __restrict__ grad,
    int64_t mlp_off, double* __restrict__ loss, int* __restrict__ status, const float2* __restrict__ enc) {
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int KH = KMAX / 2;
    const int g = G > 1 ? (int)warp_uniform(threadIdx.x >> 8) : 0;
    const int t = G > 1 ? (int)(threadIdx.x & 255) : (int)threadIdx.x;
    const int warp = (int)warp_uniform((uint32_t)t >> 5), row = t & (kTile - 1), half = warp >> 2;
    uint8_t* tiles = smem + g * tt.g_bytes;
    float4* xch = reinterpret_cast<float4*>(smem + tt.x_off) + g * 2 * kTile;  // [2][kTile] partial log-sum-exps
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + tt.bar_off);  // weights, weight gradients, MMAs of each group
    DwTurn* turn = reinterpret_cast<DwTurn*>(bars + 2 + G);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(turn + 1);
    const uint32_t bar_w = smem_u32(&bars[0]), bar_dw = smem_u32(&bars[1]), bar_mma = smem_u32(&bars[2 + g]);
    const DevCfg& cfg = tc.base;
    const int L = cfg.n_layers;
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(tt.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const uint32_t wbytes = 2u * tc.w_bytes;
    if (threadIdx.x == 32) {
        for (int i = 0; i < 2 + G; ++i) mbar_init(smem_u32(&bars[i]), 1);
        turn->taken = turn->batches = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_w), "r"(wbytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(smem + tt.w_off)),
                     "l"(wblob), "r"(wbytes), "r"(bar_w)
                     : "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tslot);
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    {
        // The weight-gradient accumulators start at zero.
        const uint32_t z[8] = {};
        for (uint32_t c = 8u * (threadIdx.x >> 7); c < tt.acc_col; c += 8u * (kTrainThreads * G / 128)) tmem_st(tmem + lanes + c, z);
        tmem_wait_st();
        tc_fence_before();
    }
    bool ok = !__syncthreads_or(threadIdx.x < 32 && !mbar_wait_bounded(bar_w, 0));
    tc_fence_after();
    if (G == 1) grid_dep_launch();  // (two groups: 593 -> 600 us with it)
    uint32_t phase = 0;
    bool issued = false;
    const uint32_t acc = tmem + tt.acc_col + (uint32_t)g * tt.acc_cols;
    const uint32_t park = tmem + tt.park_col + 32u * (uint32_t)g + 16u * (uint32_t)half + lanes;
    const uint32_t sW_addr = smem_u32(smem + tt.w_off), tile_addr = smem_u32(tiles);
    const uint32_t wlo = tc.w_bytes;  // residual weights follow the high parts
    // Grid levels of this half: [lv0, lv1); the second half also encodes the
    // product-mode inputs and the padding.
    const int nl0 = (cfg.n_levels + 1) / 2;
    const int lv0 = half ? nl0 : 0, lv1 = half ? cfg.n_levels : nl0;
    float lacc = 0.0f;
    // Deferred grid scatter (2-feature grids): a tile's encoder gradient of
    // this thread's eight levels waits in tensor memory for the next tile,
    // whose MMA waits each issue one level's atomics: the L2 atomics then
    // overlap the tensor-core work instead of following it. The warp that
    // issues a layer's MMAs (1,000 to 2,400 cycles) leaves its level for later
    // and another warp issues the next layer's, so that the group's barrier
    // does not wait for one warp's MMAs and atomics (product-mode network,
    // 2^19 samples, training step 602 -> 594 us).
    float px = 0.0f, py = 0.0f, pz = 0.0f;
    bool pend = false, pvalid = false;
    int pq = 0;  // pending levels already issued
    auto scatter_next = [&]() {
        if (F2 && pend && pq < 8) {
            uint32_t r[2];
            __syncwarp();
            tmem_ld2(park + 2u * (uint32_t)pq, r);
            tmem_wait2(r);
            const int l = 8 * half + pq;
            if (pvalid && l < cfg.n_levels) {
                const Cell cl = make_cell(px, py, pz, cfg.level_res[l]);
                float* gl = grad + (size_t)cfg.level_off[l] * 2;
                uint32_t idx[8];
                float ws[8];
                corners8(cfg, l, cl, idx, ws);
#pragma unroll
                for (int c = 0; c < 8; c += 2)
                    scatter_pair2(gl, cfg.level_off[l] + cfg.grid_shift, idx[c], idx[c + 1], ws[c], ws[c + 1],
                                  __uint_as_float(r[0]), __uint_as_float(r[1]));
            }
            __syncwarp();
            ++pq;
        }
    };
    // Waits for this group's MMAs; a wait that gives up is made known to the
    // group at its next barrier.
    auto wait_mma = [&]() {
        ok = __all_sync(0xffffffffu, ok && mbar_wait_bounded(bar_mma, phase));
        phase ^= 1u;
        tc_fence_after();
    };
    const int64_t ntiles = (n + kTile - 1) / kTile;
    // (a wait that gave up ends the loop at the group's next barrier, for all)
    for (int64_t tile = blockIdx.x + (int64_t)g * gridDim.x; tile < ntiles; tile += (int64_t)gridDim.x * G) {
        const int64_t j = tile * kTile + row;
        const bool valid = j < n;
        uint8_t* rest = tiles + tt.slot[L];
        if (F2 && enc) {
            // This half's grid features (k_train_encode), then the
            // product-mode inputs and the padding.
            float2 ev[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                ev[q] = (valid && lv0 + q < lv1) ? __ldg(enc + (int64_t)(lv0 + q) * n + j) : make_float2(0.0f, 0.0f);
            tc_encode<F2>(tc, grid32, j, valid, ld, pos, aux, tiles, row, tt.slot[L], lv1, lv1, half == 1);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (lv0 + q < lv1) store_pair(tiles, plane_off(row, 2 * (lv0 + q)), ev[q].x, ev[q].y, tt.slot[L]);
        } else {
            tc_encode<F2>(tc, grid32, j, valid, ld, pos, aux, tiles, row, tt.slot[L], lv0, lv1, half == 1);
        }
        // The loss inputs of this row, loaded now so that their latency
        // passes during the forward layers' tensor-core round trips.
        float w[3] = {0.0f, 0.0f, 1.0f}, sc = 0.0f;
        if (valid) {
            w[0] = dir[j];
            w[1] = dir[ld + j];
            w[2] = dir[2 * ld + j];
            sc = dlogv ? dlogv[j] : -(rad[j] / spdf[j]) * inv_n;
        }
        fence_async_smem();
        tc_fence_before();
        if (train_sync_or(g, !ok)) {
            ok = false;
            break;
        }
        float raw[4 * KH];
        // Forward, keeping every layer's input tile.
        for (int l = 0; l < L; ++l) {
            const TcLayer& ly = tc.layer[l];
            const bool issuer = warp == (F2 ? l & 7 : 0);
            if (issuer) {
                tc_fence_after();
                // K step s starts two planes (256 units of 16 bytes) further.
                const uint32_t sbo = (uint32_t)(ly.Kp >> 3) * 128u;
                const uint64_t ad0 = umma_desc(tile_addr + tt.slot[l], kPlane, 128u);
                const uint64_t al0 = umma_desc(tile_addr + tt.slot[L], kPlane, 128u);
                const uint64_t bd0 = umma_desc(sW_addr + ly.w_off, 128u, sbo);
                const uint64_t bl0 = umma_desc(sW_addr + wlo + ly.w_off, 128u, sbo);
                if (elect_one()) {
                    for (int s = 0; s < (ly.Kp >> 4); ++s) {
                        const uint64_t oa = (uint64_t)(256 * s), ob = (uint64_t)(16 * s);
                        mma_bf16(acc, ad0 + oa, bd0 + ob, ly.idesc, s > 0 ? 1u : 0u);
                        mma_bf16(acc, ad0 + oa, bl0 + ob, ly.idesc, 1u);
                        mma_bf16(acc, al0 + oa, bd0 + ob, ly.idesc, 1u);
                    }
                    mma_commit(bar_mma);
                }
                __syncwarp();
                issued = true;
            } else {
                scatter_next();  // the previous tile's grid gradient, one level
                if (F2) issued = true;  // (by any warp)
            }
            wait_mma();
            if (l < L - 1) {
                if (ok) {
                    uint8_t* hn = tiles + tt.slot[l + 1];
                    const uint32_t lo = tt.slot[L] - tt.slot[l + 1];
                    for (int c0 = 16 * half; c0 < ly.Np; c0 += 32) {
                        uint32_t r[16];
                        tmem_ld16(acc + lanes + (uint32_t)c0, r);
                        tmem_wait16(r);
                        float v[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = fmaxf(__uint_as_float(r[i]), 0.0f);
                        store_cols<16>(hn, row, c0, v, lo);
                    }
                }
                fence_async_smem();
                tc_fence_before();
                if (train_sync_or(g, !ok)) {
                    ok = false;
                    break;
                }
            } else if (ok) {
                // This half's lobes: columns [half * 4 KH, (half + 1) * 4 KH).
                if constexpr (4 * KH >= 16) {
#pragma unroll
                    for (int c = 0; c < 4 * KH / 16; ++c) {
                        uint32_t r[16] = {};
                        if (half * 4 * KH + 16 * c < ly.Np) {
                            tmem_ld16(acc + lanes + (uint32_t)(half * 4 * KH + 16 * c), r);
                            tmem_wait16(r);
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i) raw[16 * c + i] = __uint_as_float(r[i]);
                    }
                } else {
                    uint32_t r[16];
                    tmem_ld16(acc + lanes, r);
                    tmem_wait16(r);
#pragma unroll
                    for (int i = 0; i < 4 * KH; ++i) raw[i] = __uint_as_float(half ? r[4 * KH + i] : r[i]);
                }
            }
        }
        // Loss and d loss / d raw (zero for rows beyond n).
        {
            GradHalf<KMAX> gh;
            float4 part = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (ok) part = gh.pass1(cfg, half, raw, w);
            xch[half * kTile + row] = part;
            if (train_sync_or(g, !ok)) {
                ok = false;
                break;
            }
            const float4 oth = xch[(half ^ 1) * kTile + row];
            const float lse = lse_combine(part.x, part.y, oth.x, oth.y);
            const float lsa = lse_combine(part.z, part.w, oth.z, oth.w);
            if (valid && half == 0) lacc += sc * (lsa - lse);
            float dr[4 * KH];
            gh.pass2(lse, lsa, sc, dr);
            // (columns beyond the last layer's padded outputs do not exist)
            if constexpr (4 * KH >= 16) {
#pragma unroll
                for (int c = 0; c < 4 * KH; c += 16)
                    if (half * 4 * KH + c < tc.layer[L - 1].Np)
                        store_cols<16>(rest, row, half * 4 * KH + c, dr + c, (uint32_t)tc.layer[L - 1].Np * (kPlane / 8));
            } else {
                store_cols<4 * KH>(rest, row, half * 4 * KH, dr, (uint32_t)tc.layer[L - 1].Np * (kPlane / 8));
            }
        }
        fence_async_smem();
        tc_fence_before();
        train_sync(g);
        // Backward, top layer first.
        for (int l = L - 1; l >= 0; --l) {
            const TcLayer& ly = tc.layer[l];
            const uint32_t lo_off = (uint32_t)ly.Np * (kPlane / 8);  // residuals behind the output gradient
            const bool issuer = warp == (F2 ? (2 * L - 1 - l) & 7 : 0);
            if (issuer) {
                tc_fence_after();
                const uint32_t hk = (uint32_t)(ly.Kp >> 3) * 128u;  // K step of a W_l tile
                const uint32_t d_addr = tile_addr + tt.slot[l + 1];
                // D W_l: M = 128 samples, N = Kp_l, K = Np_l outputs.
                const uint64_t ad0 = umma_desc(d_addr, kPlane, 128u), al0 = umma_desc(d_addr + lo_off, kPlane, 128u);
                const uint64_t bd0 = umma_desc(sW_addr + ly.w_off, hk, 128u);
                const uint64_t bl0 = umma_desc(sW_addr + wlo + ly.w_off, hk, 128u);
                const uint64_t bstep = (uint64_t)((2u * hk) >> 4);
                // dW_l += D^T H_l: M = 128 (outputs, then their residuals),
                // N = Kp_l, K = 128 samples (256 bytes a step).
                const uint64_t bh0 = umma_desc(tile_addr + tt.slot[l], 128u, kPlane);
                const uint64_t dw0 = umma_desc(d_addr, 128u, kPlane), dwl0 = umma_desc(d_addr + lo_off, 128u, kPlane);
                if (elect_one()) {
                    for (int s = 0; s < (ly.Np >> 4); ++s) {
                        const uint64_t oa = (uint64_t)(256 * s), ob = s * bstep;
                        mma_bf16(acc, ad0 + oa, bd0 + ob, tt.idesc_dx[l], s > 0 ? 1u : 0u);
                        mma_bf16(acc, ad0 + oa, bl0 + ob, tt.idesc_dx[l], 1u);
                        mma_bf16(acc, al0 + oa, bd0 + ob, tt.idesc_dx[l], 1u);
                    }
                    if (G == 1 || take_turn(turn, bar_dw)) {
                        tc_fence_after();
                        for (int s = 0; s < 8; ++s) {
                            const uint64_t o = (uint64_t)(16 * s);
                            mma_bf16(tmem + tt.dw_col[l], dw0 + o, bh0 + o, tt.idesc_dw[l], 1u);
                            if (2 * ly.Np > 128) mma_bf16(tmem + tt.dw_col[l], dwl0 + o, bh0 + o, tt.idesc_dw[l], 1u);
                        }
                        if (G > 1) {
                            mma_commit(bar_dw);
                            pass_turn(turn);
                        }
                    } else {
                        ok = false;
                    }
                    mma_commit(bar_mma);
                }
                __syncwarp();
            } else {
                scatter_next();
            }
            wait_mma();
            if (l > 0) {
                // The gradient of layer l's input, D W_l where the input is
                // positive (ReLU'), in its place.
                if (ok) {
                    uint8_t* hl = tiles + tt.slot[l];
                    for (int c0 = 16 * half; c0 < ly.Kp; c0 += 32) {
                        uint32_t r[16];
                        tmem_ld16(acc + lanes + (uint32_t)c0, r);
                        tmem_wait16(r);
                        const uint4 m0 = *reinterpret_cast<const uint4*>(hl + plane_off(row, c0));
                        const uint4 m1 = *reinterpret_cast<const uint4*>(hl + plane_off(row, c0 + 8));
                        const uint32_t mw[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                        float v[16];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float2 hv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&mw[i]));
                            v[2 * i] = hv.x > 0.0f ? __uint_as_float(r[2 * i]) : 0.0f;
                            v[2 * i + 1] = hv.y > 0.0f ? __uint_as_float(r[2 * i + 1]) : 0.0f;
                        }
                        store_cols<16>(hl, row, c0, v, (uint32_t)ly.Kp * (kPlane / 8));
                    }
                }
                fence_async_smem();
                tc_fence_before();
                if (train_sync_or(g, !ok)) {
                    ok = false;
                    break;
                }
            } else if (ok && 16 * half < cfg.grid_feats) {
                // Encoder gradient of this half's 16 grid-feature columns ->
                // grid scatter.
                uint32_t r[16];
                tmem_ld16(acc + lanes + (uint32_t)(16 * half), r);
                tmem_wait16(r);
                if (F2 && tt.park) {
                    while (pend && pq < 8) scatter_next();  // what the layers left
                    const uint32_t a[8] = {r[0], r[1], r[2], r[3], r[4], r[5], r[6], r[7]};
                    const uint32_t b[8] = {r[8], r[9], r[10], r[11], r[12], r[13], r[14], r[15]};
                    tmem_st(park, a);
                    tmem_st(park + 8u, b);
                    tmem_wait_st();
                    pend = true;
                    pvalid = valid;
                    pq = 0;
                    if (valid) {
                        px = pos[j];
                        py = pos[ld + j];
                        pz = pos[2 * ld + j];
                    }
                } else if (valid) {
                    float dg[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) dg[i] = __uint_as_float(r[i]);
                    const float x = pos[j], y = pos[ld + j], z = pos[2 * ld + j];
                    const int F = cfg.feat;
                    if (F == 2) scatter_levels<2, 8>(cfg, grad, x, y, z, 8 * half, dg);
                    else if (F == 4) scatter_levels<4, 4>(cfg, grad, x, y, z, 4 * half, dg);
                    else if (F == 8) scatter_levels<8, 2>(cfg, grad, x, y, z, 2 * half, dg);
                    else scatter_levels<1, 16>(cfg, grad, x, y, z, 16 * half, dg);
                }
                __syncwarp();
                tc_fence_before();
            } else {
                tc_fence_before();
            }
        }
    }
    while (pend && pq < 8) scatter_next();  // the last tile's grid gradient
    // Loss: one atomic per warp.
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
    if (loss && (t & 31) == 0 && lacc != 0.0f) atomicAdd(loss, (double)lacc);
    if (!ok) {
        if ((t & 31) == 0) atomicOr(status, kStatusTimeout);
        // Before the tensor memory is released: wait again, bounded, for this
        // group's MMAs that may still be in flight.
        if (t == 0 && issued) (void)mbar_wait_bounded(bar_mma, phase ^ 1u);
    }
    // Weight gradients, once every group is done: lane o of layer l's columns
    // holds D_hi^T H, lane Np + o the residuals' share (or the lane of the high
    // part both). The shares meet in shared memory (the tiles are done with),
    // and four weights leave in one operation: every CTA adds to the same few
    // kilobytes, whose L2 slices take the operations one after another (with
    // one per weight and share that was two thirds of the small network's
    // kernel).
    tc_fence_before();
    const bool all_ok = !__syncthreads_or(!ok);
    tc_fence_after();
    if (all_ok) {
        const int lane = (int)(threadIdx.x & 127), set = (int)(threadIdx.x >> 7);
        constexpr int kSets = kTrainThreads * G / 128;
        float* stage = reinterpret_cast<float*>(smem);
        for (int pass = 0; pass < 2; ++pass) {
            float* sl = stage;
            for (int l = 0; l < L; ++l) {
                const TcLayer& ly = tc.layer[l];
                const bool both = 2 * ly.Np <= 128;
                float* gW = grad + mlp_off + tt.woff[l] + (int64_t)lane * ly.K;
                const bool wide = (reinterpret_cast<uintptr_t>(grad + mlp_off) & 15u) == 0;
                const bool mine = pass == 0 ? both && lane >= ly.Np && lane < 2 * ly.Np : lane < ly.N;
                for (int c0 = 16 * set; c0 < ly.Kp; c0 += 16 * kSets) {
                    uint32_t r[16];
                    tmem_ld16(tmem + lanes + tt.dw_col[l] + (uint32_t)c0, r);
                    tmem_wait16(r);
                    if (mine) {
                        // stage: [Kp / 4][Np] vectors, so that a warp's lie side by side
#pragma unroll
                        for (int i = 0; i < 16; i += 4) {
                            float4* st4 = reinterpret_cast<float4*>(sl) + (size_t)((c0 + i) >> 2) * ly.Np;
                            float4 v = make_float4(__uint_as_float(r[i]), __uint_as_float(r[i + 1]),
                                                   __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
                            if (pass == 0) {
                                st4[lane - ly.Np] = v;
                            } else if (c0 + i < ly.K) {
                                if (both) {
                                    const float4 lo = st4[lane];
                                    v = make_float4(v.x + lo.x, v.y + lo.y, v.z + lo.z, v.w + lo.w);
                                }
                                red_add4(gW + c0 + i, wide, v.x, v.y, v.z, v.w);
                            }
                        }
                    }
                    __syncwarp();
                }
                if (both) sl += ly.Kp * ly.Np;
            }
            __syncthreads();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tt.tmem_cols) : "memory");
    }
}

}  // namespace

struct TcState {
    TcCfg cfg;
    uint8_t* wblob = nullptr;      // BF16 weights of the training parameters
    // Training always multiplies split operands (BF16 high part and
    // residual): with single-pass BF16 inference (NPM_BF16) this is a second
    // blob in the split layout; otherwise training reads wblob.
    uint8_t* wblob_train = nullptr;
    uint8_t* wblob_inf = nullptr;  // of the moving average, when inference uses it
    TcCfg train_cfg;     // copy of cfg for training (split operands)
    TcTrain train;
    bool can_train = false;
    // Corner blocks of the inference table (npm_tc.cuh), the version of the
    // parameters that each chunk was built from, and their number; NULL: none
    // (a handle whose batches cannot be large enough to use them).
    uint4* blk = nullptr;
    int* blk_built = nullptr;
    uint32_t blk_total = 0;
    // Grid features of a training batch (max_batch x grid_feats FP32) for
    // 2-feature grids, written by k_train_encode; NULL: the training kernel
    // gathers them itself.
    float2* enc = nullptr;
};

static int pad16(int v) { return (v + 15) / 16 * 16; }

npm_status tc_create(npm_handle* h) {
    const npm_config& c = h->cfg;
    const bool fp32 = c.precision == NPM_FP32;
    if (!fp32 && c.feat_per_level != 1 && c.feat_per_level != 2 && c.feat_per_level != 4 &&
        c.feat_per_level != 8)
        return NPM_ERR_UNSUPPORTED;
    TcState* s = new TcState();
    TcCfg& t = s->cfg;
    memset(&t, 0, sizeof(t));
    t.base = h->dc;
    uint32_t off = 0;
    int maxnp = 0;
    for (int l = 0; l < c.n_layers; ++l) {
        TcLayer& ly = t.layer[l];
        ly.K = c.widths[l];
        ly.N = c.widths[l + 1];
        ly.Kp = pad16(ly.K);
        ly.Np = pad16(ly.N);
        ly.w_off = off;
        off += (uint32_t)(ly.Np * ly.Kp * 2);
        // kind::f16 descriptor: D FP32 (bit 4), A and B BF16 (bits 7, 10;
        // zero for FP16 operands), both K-major, N >> 3 at bit 17, M >> 4 at
        // bit 24.
        const bool f16ops = c.precision == NPM_FP16 || c.precision == NPM_FP32_TC;
        const uint32_t ab = f16ops ? 0u : (1u << 7) | (1u << 10);
        ly.idesc = (1u << 4) | ab | ((uint32_t)(ly.Np >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
        maxnp = ly.Np > maxnp ? ly.Np : maxnp;
    }
    t.w_bytes = (off + 127u) / 128u * 128u;
    t.split = (c.precision == NPM_BF16X3 || c.precision == NPM_FP32_TC) ? 1 : 0;
    t.f16 = (c.precision == NPM_FP16 || c.precision == NPM_FP32_TC) ? 1 : 0;
    t.fp32 = (c.precision == NPM_FP32_TC || fp32) ? 1 : 0;
    t.parts = fp32 ? 3 : t.split ? 2 : 1;
    t.wparts = fp32 ? 3 : (t.split || t.f16) ? 2 : 1;
    const uint32_t nsplit = (uint32_t)t.parts, nw = (uint32_t)t.wparts;
    int maxkp = 16;
    for (int l = 0; l < c.n_layers; ++l) maxkp = std::max(maxkp, t.layer[l].Kp);
    t.d_cols = (uint32_t)((maxnp + 31) / 32 * 32);
    t.a_cols = (uint32_t)(maxkp / 2);
    // FP32 models that do not fit keep the CUDA-core kernels. In the other
    // modes the limit is part of the interface: 200 KB for the weights and one
    // activation tile per part (two where the encoding leaves whole 8-column
    // chunks of a multi-level network's first layer empty).
    const int enc_width = c.n_levels * c.feat_per_level + (c.mode == NPM_PRODUCT ? 21 : 0);
    const bool one_level = c.n_levels == 1 && c.feat_per_level <= 8 && c.mode != NPM_PRODUCT;
    const bool sep0 = (enc_width + 7) / 8 * 8 < t.layer[0].Kp && !one_level;
    int hidden = 16;  // widest input of the layers that share a tile
    for (int l = sep0 ? 1 : 0; l < c.n_layers; ++l) hidden = std::max(hidden, t.layer[l].Kp);
    const uint32_t tile_bytes = (uint32_t)(kTile * (hidden + (sep0 ? t.layer[0].Kp : 0)) * 2);
    if (fp32 ? nw * t.w_bytes + (uint32_t)(kTile * maxkp * 2) > 224 * 1024
             : nw * t.w_bytes + nsplit * tile_bytes + 64 > 200 * 1024 || c.K > 16) {
        delete s;
        return NPM_ERR_UNSUPPORTED;
    }
    // Training layout. Gradients take split BF16 operands in every
    // reduced-precision mode: single-pass BF16 compounds its rounding down
    // the layers and through the cancelling grid sums (per-tensor gradient
    // errors of tens of percent), so only inference offers the plain form.
    {
        TcTrain& tr = s->train;
        memset(&tr, 0, sizeof(tr));
        s->train_cfg = t;
        // Training multiplies BF16 operands whatever the inference format.
        s->train_cfg.f16 = 0;
        s->train_cfg.split = 1;
        s->train_cfg.wparts = 2;
        for (int l = 0; l < c.n_layers; ++l) s->train_cfg.layer[l].idesc |= (1u << 7) | (1u << 10);
        uint32_t off = 0, cols = 0;
        int64_t wo = 0;
        int wide = 16, maxin = 16;  // widest layer, widest input
        bool fits = c.K * 4 <= 64 && c.n_levels * c.feat_per_level <= 32;
        for (int l = 0; l < c.n_layers; ++l) {
            const TcLayer& ly = t.layer[l];
            tr.slot[l] = off;
            off += (uint32_t)(kTile * ly.Kp * 2);
            maxin = std::max(maxin, ly.Kp);
            wide = std::max(wide, std::max(ly.Kp, ly.Np));
            tr.woff[l] = wo;
            wo += (int64_t)ly.K * ly.N;
            if (ly.Np > 128 || ly.Kp > 128) fits = false;
            tr.dw_col[l] = cols;
            cols += (uint32_t)ly.Kp;
            // dW: A = delta^T (MN-major), B = H_l (MN-major), M = 128, N = Kp_l.
            tr.idesc_dw[l] = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                             ((uint32_t)(ly.Kp >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
            // dX: A = delta (K-major), B = W_l read MN-major, M = 128, N = Kp_l.
            tr.idesc_dx[l] = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) |
                             ((uint32_t)(ly.Kp >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
        }
        // Which networks train on tensor cores is part of the interface: those
        // whose weights, tiles and a gradient tile pair as wide as the widest
        // layer fit 220 KB, with the accumulators in 512 columns. This layout
        // is never larger.
        const uint32_t need = 2u * t.w_bytes + off + 2u * kTile * wide * 2u + kTile * maxin * 2u + 64u;
        uint32_t pw = 32;
        while (pw < cols + (uint32_t)wide) pw <<= 1;
        // FP32 and the FP32-accuracy mode train with the FP32 kernels.
        s->can_train = fits && pw <= 512 && need <= 220 * 1024 && !t.fp32;
        const int last = t.layer[c.n_layers - 1].Np;
        tr.slot[c.n_layers] = off;
        off += (uint32_t)(kTile * std::max(maxin, 2 * last) * 2);
        tr.g_bytes = off;
        tr.acc_col = cols;
        tr.acc_cols = (uint32_t)wide;
        // Two groups where they fit; sixteen lobes take the registers of one.
        // Networks of up to four lobes on grids without 2 features run the
        // instance of one group and three CTAs an SM instead, whatever their
        // layers' widths: measured on the small network alone, for which it was
        // made, and not on wide layers of which fewer CTAs fit.
        auto lay = [&](int G) {
            tr.groups = G;
            tr.x_off = (uint32_t)G * tr.g_bytes;
            tr.w_off = tr.x_off + (uint32_t)G * 2u * kTile * 16u;
            // An MMA reads 128 rows from the start of a gradient's slot.
            uint32_t end = tr.w_off + 2u * t.w_bytes;
            for (int l = 1; l <= c.n_layers; ++l)
                end = std::max(end, (uint32_t)(G - 1) * tr.g_bytes + tr.slot[l] + 16u * kPlane +
                                        (2 * t.layer[l - 1].Np > 128 ? (uint32_t)t.layer[l - 1].Np * (kPlane / 8) : 0u));
            tr.bar_off = (end + 127u) / 128u * 128u;
            tr.smem = tr.bar_off + 8u * (2u + (uint32_t)G) + 32u;
            uint32_t used = cols + (uint32_t)G * (uint32_t)wide;
            tr.park = c.feat_per_level == 2 && used + 32u * (uint32_t)G <= 512u ? 1 : 0;
            tr.park_col = used;
            if (tr.park) used += 32u * (uint32_t)G;
            tr.tmem_cols = 32;
            while (tr.tmem_cols < used) tr.tmem_cols <<= 1;
            return tr.tmem_cols <= 512u && tr.smem <= 227u * 1024u;
        };
        const bool small = c.K <= 4 && c.feat_per_level != 2;
        if (small || c.K > 8 || !lay(2)) {
            if (!lay(1)) s->can_train = false;
        }
    }
    if (device_alloc((void**)&s->wblob, nw * t.w_bytes) != cudaSuccess) {
        cudaGetLastError();
        delete s;
        return NPM_ERR_OOM;
    }
    cudaMemset(s->wblob, 0, nw * t.w_bytes);
    if (s->can_train && !t.split) {
        if (device_alloc((void**)&s->wblob_train, 2u * t.w_bytes) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(s->wblob);
            delete s;
            return NPM_ERR_OOM;
        }
        cudaMemset(s->wblob_train, 0, 2u * t.w_bytes);
    }
    if (s->can_train && c.feat_per_level == 2) {
        // Optional: without it the training kernel encodes in place.
        if (device_alloc((void**)&s->enc, sizeof(float) * (size_t)c.max_batch * h->dc.grid_feats) != cudaSuccess) {
            cudaGetLastError();
            s->enc = nullptr;
        }
    }
    // Corner blocks, in level order while they stay a part of the L2 (64 of 129
    // MB).
    if ((c.feat_per_level == 2 || c.feat_per_level == 4) && !tiny_qualifies(t)) {  // (that keeps its table in shared memory)
        constexpr uint64_t kMost = (64ull << 20) / 32;
        uint64_t total = 0;
        for (int l = 0; l < c.n_levels; ++l) {
            const uint64_t D = (uint64_t)c.level_res[l], entries = D * D * D;
            if (!((h->dc.dense_mask >> l) & 1u) || total + entries > kMost) continue;
            t.blk_mask |= 1u << l;
            t.blk_off[l] = (uint32_t)total;
            total += entries;
        }
        s->blk_total = (uint32_t)total;
    }
    h->tc = s;
    tc_reserve_blocks(h, c.max_batch);
    return NPM_OK;
}

void tc_reserve_blocks(npm_handle* h, int64_t queries) {
    TcState* s = h->tc;
    if (!s || s->blk || !s->blk_total || queries < kBlkMinQueries) return;
    const size_t chunks = (s->blk_total + kBlkChunk - 1) / kBlkChunk;
    uint4* blk = nullptr;
    int* built = nullptr;
    // Optional: without them large batches read the table too.
    if (device_alloc((void**)&blk, 32 * (size_t)s->blk_total) == cudaSuccess &&
        device_alloc((void**)&built, chunks * sizeof(int)) == cudaSuccess &&
        cudaMemset(built, 0, chunks * sizeof(int)) == cudaSuccess && cudaStreamSynchronize(0) == cudaSuccess) {
        s->blk = blk;
        s->blk_built = built;
        return;
    }
    cudaGetLastError();
    if (blk) cudaFree(blk);
    if (built) cudaFree(built);
}

void tc_destroy(npm_handle* h) {
    if (!h->tc) return;
    if (h->tc->wblob) cudaFree(h->tc->wblob);
    if (h->tc->wblob_inf) cudaFree(h->tc->wblob_inf);
    if (h->tc->wblob_train) cudaFree(h->tc->wblob_train);
    if (h->tc->enc) cudaFree(h->tc->enc);
    if (h->tc->blk) cudaFree(h->tc->blk);
    if (h->tc->blk_built) cudaFree(h->tc->blk_built);
    delete h->tc;
    h->tc = nullptr;
}

cudaError_t tc_refresh_weights(npm_handle* h, bool cuda_cores, const UpdateEnd& end, cudaStream_t st) {
    TcState* s = h->tc;
    // The launch that ends the update comes last.
    auto arrange = [&](const TcCfg& cfg, const float* mlp, uint8_t* blob, float* wfwd, const UpdateEnd& e) {
        return launch_maybe_pdl(k_tc_weights, dim3(16, h->dc.n_layers), dim3(256), 0, st, true, cfg, mlp, blob, wfwd, e);
    };
    cudaError_t e = cudaSuccess;
    if (s->wblob_train)
        e = arrange(s->train_cfg, h->params + h->mlp_off, s->wblob_train, nullptr, UpdateEnd{});
    if (e == cudaSuccess && h->ema) {
        if (!s->wblob_inf) {
            const size_t bytes = (size_t)s->cfg.wparts * s->cfg.w_bytes;
            e = cudaMalloc(&s->wblob_inf, bytes);
            if (e != cudaSuccess) return e;
            cudaMemsetAsync(s->wblob_inf, 0, bytes, st);
        }
        e = arrange(s->cfg, h->ema + h->mlp_off, s->wblob_inf, nullptr, UpdateEnd{});
    }
    if (e != cudaSuccess) return e;
    return arrange(s->cfg, h->params + h->mlp_off, s->wblob, cuda_cores ? h->wfwd : nullptr, end);
}

template <int KMAX, bool F2, int G>
static cudaError_t launch_train_tc(npm_handle* h, int64_t n, int64_t ld, const float* pos, const float* aux,
                                   const float* dir, const float* rad, const float* spdf, const float* dlogv,
                                   double* loss, cudaStream_t st) {
    TcState* s = h->tc;
    auto kern = k_train_tc<KMAX, F2, G>;
    // CTAs per SM: the instance's register budget, if shared and tensor
    // memory hold that many.
    int per_sm = train_ctas_per_sm(KMAX, F2, G);
    while (per_sm > 1 && ((size_t)per_sm * (s->train.smem + 1024) > 227 * 1024 ||
                          (uint32_t)per_sm * s->train.tmem_cols > 512u))
        --per_sm;
    static std::atomic<uint64_t> attrs{~0ull};
    cudaError_t e =
        set_smem_attrs(kern, s->train.smem, carveout_percent((size_t)per_sm * (s->train.smem + 1024)), attrs);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ntiles = (n + kTile - 1) / kTile;
    const int64_t slots = (int64_t)per_sm * sms;
    const int g = (int)(ntiles < slots ? ntiles : slots);
    int* status = reinterpret_cast<int*>(h->scalars + 8);
    const float2* enc = nullptr;
    if (F2 && s->enc && n <= h->cfg.max_batch) {
        const dim3 grid((unsigned)((n + 255) / 256), (unsigned)((h->dc.n_levels + kEncLevels - 1) / kEncLevels));
        k_train_encode<<<grid, 256, 0, st>>>(h->dc, h->params, n, ld, pos, s->enc);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        enc = s->enc;
    }
    const uint8_t* wb = s->wblob_train ? s->wblob_train : s->wblob;
    kern<<<g < 1 ? 1 : g, kTrainThreads * G, s->train.smem, st>>>(s->train_cfg, s->train, h->params, wb, n, ld, pos,
                                                                  aux, dir, rad, spdf, dlogv, 1.0f / (float)n,
                                                                  h->grads, h->mlp_off, loss, status, enc);
    return cudaGetLastError();
}

bool tc_can_train(npm_handle* h) { return h->tc && h->tc->can_train; }

cudaError_t tc_train(npm_handle* h, int64_t n, int64_t ld, const float* pos, const float* aux, const float* dir,
                     const float* rad, const float* spdf, const float* dlogv, double* loss, cudaStream_t st) {
    const int K = h->cfg.K;
    const bool f2 = h->cfg.feat_per_level == 2;
    const bool two = h->tc->train.groups == 2;
    if (K <= 4 && !f2) return launch_train_tc<4, false, 1>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st);
    if (K <= 8) {
        if (f2)
            return two ? launch_train_tc<8, true, 2>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st)
                       : launch_train_tc<8, true, 1>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st);
        return two ? launch_train_tc<8, false, 2>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st)
                   : launch_train_tc<8, false, 1>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st);
    }
    return f2 ? launch_train_tc<16, true, 1>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st)
              : launch_train_tc<16, false, 1>(h, n, ld, pos, aux, dir, rad, spdf, dlogv, loss, st);
}

// The corner blocks of the inference table, brought up to date on st.
template <typename GT>
static cudaError_t update_blocks(npm_handle* h, const GT* table, const int* shared, cudaStream_t st) {
    TcState* s = h->tc;
    const unsigned chunks = (s->blk_total + kBlkChunk - 1) / kBlkChunk;
    if (h->cfg.feat_per_level == 2)
        k_corner_blocks<GT, 2><<<chunks, 256, 0, st>>>(s->cfg, table, s->blk, s->blk_total, s->blk_built,
                                                       version_word(h), shared);
    else
        k_corner_blocks<GT, 4><<<chunks, 256, 0, st>>>(s->cfg, table, s->blk, s->blk_total, s->blk_built,
                                                       version_word(h), shared);
    return cudaGetLastError();
}

cudaError_t tc_query_batch(npm_handle* h, QueryBatch& qb, int64_t max_n, cudaStream_t st, bool pdl) {
    const TcState* s = h->tc;
    const TcCfg& c = s->cfg;
    const uint8_t* wb = h->ema ? s->wblob_inf : s->wblob;  // inference weights
    int* status = status_word(h);
    // The small serving networks get their own kernel (npm_tc_tiny.cu);
    // tuning override NPM_TC_TINY=0 selects the general kernel instead.
    static std::atomic<int> env_tiny{INT32_MIN + 1};
    if (tiny_qualifies(c) && env_override("NPM_TC_TINY", env_tiny) != 0)
        return launch_tiny(c, h->grid_h, wb, qb, max_n, status, st, pdl);
    // Large batches read the dense levels through corner blocks.
    int64_t queries = 0;
    for (int i = 0; i < qb.nseg; ++i) queries += qb.seg[i].n;
    if (qb.n_dev) queries = max_n;
    const uint4* blk = s->blk && queries >= kBlkMinQueries ? s->blk : nullptr;
    if (blk) {
        // FP32 tables are the parameters themselves: a caller that holds
        // their address may change them unseen. The flag is read on the
        // device: a graph may be captured before the address is handed out.
        cudaError_t e = c.fp32 ? update_blocks(h, inf_params(h), shared_word(h), st)
                               : update_blocks(h, h->grid_h, nullptr, st);
        if (e != cudaSuccess) return e;
    }
    const long long limit = 1ll << 32;  // the 16-bit kernels' fixed bound
    // FP32 and the FP32-accuracy mode gather from the FP32 table.
    if (c.parts == 3)
        return launch_fwd_ops<kThreeBf16>(c, inf_params(h), blk, wb, qb, max_n, status, h->wait_limit, false, st);
    if (c.fp32) return launch_fwd_ops<kTwoFp16>(c, inf_params(h), blk, wb, qb, max_n, status, limit, false, st);
    // Tuning override NPM_TC_DECODE=1: the warp-per-query decode (up to eight
    // lobes).
    static std::atomic<int> env_dec{INT32_MIN + 1};
    const bool warp_decode = c.base.K <= 8 && env_override("NPM_TC_DECODE", env_dec) == 1;
    if (c.f16) return launch_fwd_ops<kOneFp16>(c, h->grid_h, blk, wb, qb, max_n, status, limit, warp_decode, st);
    if (c.split) return launch_fwd_ops<kTwoBf16>(c, h->grid_h, blk, wb, qb, max_n, status, limit, warp_decode, st);
    return launch_fwd_ops<kOneBf16>(c, h->grid_h, blk, wb, qb, max_n, status, limit, warp_decode, st);
}

npm_status tc_query(npm_handle* h, int64_t n, int64_t ld, const float* pos, const float* aux,
                    const float* uin, float ufrac, bool sample, float* dir_out, float* pdf_out,
                    float* mix_out, cudaStream_t st, bool log_pdf) {
    QueryBatch qb;
    memset(&qb, 0, sizeof(qb));
    qb.nseg = 1;
    qb.sample = sample ? 1 : 0;
    qb.log_pdf = (!sample && log_pdf) ? 1 : 0;
    QuerySeg& q = qb.seg[0];
    q.n = n;
    q.ld = ld;
    q.pos = pos;
    q.aux = aux;
    q.uin = uin;
    q.ufrac = sample ? ufrac : 0.0f;
    q.dir = sample ? dir_out : nullptr;
    q.pdf = pdf_out;
    q.mix = sample ? mix_out : nullptr;
    return tc_query_batch(h, qb, n, st) == cudaSuccess ? NPM_OK : NPM_ERR_CUDA;
}

}  // namespace npm
