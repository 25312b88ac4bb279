// npm_fp32.cu -- FP32 CUDA-core path of the NPM hot path.
//
// Tile groups of 128 threads walk 64-query tiles. Per tile:
//   encode  : 2 threads per query gather the 8 corners of every level and
//             blend them (Sec. 5.1, Eq. 11); product mode appends the SH
//             encodings and the roughness (Sec. 4.3).
//   MLP     : each layer is a 64 x N x K tile GEMM from shared memory; thread
//             (qg, g) owns queries qg + 8j (j < 8) and outputs g*NI .. g*NI+NI-1
//             (Sec. 5.3, Eq. 12). Weights are staged once per CTA.
//   epilogue: 2 threads per query (lobes split in halves, combined with
//             warp shuffles) map the raw outputs (Table 1), then sample and/or
//             evaluate the mixture (Eq. 3-4).
// FP32 inference runs on the tensor cores in 24-bit operands
// (npm_tc_forward.cuh); this forward kernel serves the networks whose weights
// do not fit there, and the allocation-free entry point, whose scratch it
// limits to one padded copy of the weights.
// The training kernel recomputes the forward pass, forms the gradient of the
// weighted log-likelihood in the log domain (Eq. 9), back-propagates through
// the layers and scatters grid gradients with vector atomics.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <type_traits>

#include "npm_device.cuh"
#include "npm_kernels.h"

namespace npm {

constexpr int kTQ = 64;   // queries per tile
constexpr int kNT = 128;  // threads per CTA
constexpr unsigned kFull = 0xffffffffu;

// Activation row stride (floats) of the forward kernel instance whose
// widest layer is 16 * I: the padding of 4 keeps the 16 rows a warp reads
// in distinct banks.
__host__ __device__ constexpr int fwd_act_stride(int I) { return 16 * I + 4; }

// Tile groups per CTA of that instance: the register file holds 4 groups at
// 128 registers a thread, 6 at 80 (enough for the narrow instance only).
__host__ __device__ constexpr int fwd_max_groups(int I) { return I <= 2 ? 6 : 4; }

// ----------------------------------------------------------- tile GEMM

// Named barrier of tile group `group` (T threads; barrier 0 is the CTA's).
template <int T = kNT>
__device__ __forceinline__ void group_sync(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(T) : "memory");
}

template <int NI>
__device__ __forceinline__ void load_w(const float* p, float (&w)[NI]) {
    if constexpr (NI == 1) {
        w[0] = p[0];
    } else if constexpr (NI == 2) {
        float2 v = *reinterpret_cast<const float2*>(p);
        w[0] = v.x;
        w[1] = v.y;
    } else {
#pragma unroll
        for (int c = 0; c < NI; c += 4) {
            float4 v = *reinterpret_cast<const float4*>(p + c);
            w[c] = v.x;
            w[c + 1] = v.y;
            w[c + 2] = v.z;
            w[c + 3] = v.w;
        }
    }
}

// out[q][n] = f(sum_k in[q][k] * WT[k][n]) for q < 64, n < N. WT rows are
// padded to 16 * NI columns (zeros beyond N). mode 0: identity, 1: ReLU.
// AST > 0: the activation row stride is the compile-time AST (so row and
// weight addresses are immediate offsets of two pointers); else AS_rt.
// OS_rt: row stride of out (AST = 0). WPAD: floats between the weight
// rows beyond NP.
// INPLACE: out may equal in; the tile group (named barrier group + 1)
// synchronises between the last read of in and the first store.
// T: threads of the tile group; each owns 64 * 16 / T queries.
template <int NI, int AST, bool INPLACE, int WPAD = 0, int T = kNT>
__device__ __forceinline__ void tile_gemm(int t, const float* in, int AS_rt, int K,
                                          const float* __restrict__ WT, float* out, int OS_rt, int N, int mode,
                                          int group) {
    const int AS = AST > 0 ? AST : AS_rt, OS = AST > 0 ? AST : OS_rt;
    constexpr int NP = 16 * NI + WPAD;
    // Thread t owns output group g (16 groups) and query group qg (T / 16): a
    // warp covers all 16 output groups and 2 query groups, lanes 2i and
    // 2i + 1 sharing output group i. Lanes that read the same shared-memory
    // vector are adjacent, which keeps a warp's 16-byte shared loads at two
    // wavefronts (sharing between strided lanes costs four).
    const int g = (t & 31) >> 1, qg = (t & 1) | ((t >> 5) << 1);
    // Accumulators paired along adjacent outputs: one packed two-lane FMA
    // (fma.rn on each lane, the same rounding as fmaf) per pair.
    constexpr int NP2 = NI >= 2 ? NI / 2 : 1;
    constexpr int QG = T / 16, NQ = kTQ / QG;  // query groups, queries of a thread (qg + QG j)
    float2 acc[NQ][NP2];
    float acc1[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        acc1[j] = 0.0f;
#pragma unroll
        for (int i = 0; i < NP2; ++i) acc[j][i] = make_float2(0.0f, 0.0f);
    }
    if constexpr (NI <= 2) {
        // Narrow layers: the K step's 4 x NI weights stay in registers and the
        // activation rows stream through one at a time (fewer live registers,
        // so more tile groups fit).
        for (int k = 0; k < K; k += 4) {
            float w[4][NI];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) load_w<NI>(WT + (k + kk) * NP + g * NI, w[kk]);
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const float4 a = *reinterpret_cast<const float4*>(in + (qg + QG * j) * AS + k);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const float av = kk == 0 ? a.x : kk == 1 ? a.y : kk == 2 ? a.z : a.w;
                    if constexpr (NI == 1)
                        acc1[j] = fmaf(av, w[kk][0], acc1[j]);
                    else
                        acc[j][0] = __ffma2_rn(make_float2(av, av), make_float2(w[kk][0], w[kk][1]), acc[j][0]);
                }
            }
        }
    } else {
        for (int k = 0; k < K; k += 4) {
            float4 a[NQ];
#pragma unroll
            for (int j = 0; j < NQ; ++j) a[j] = *reinterpret_cast<const float4*>(in + (qg + QG * j) * AS + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                float w[NI];
                load_w<NI>(WT + (k + kk) * NP + g * NI, w);
#pragma unroll
                for (int j = 0; j < NQ; ++j) {
                    const float av = kk == 0 ? a[j].x : kk == 1 ? a[j].y : kk == 2 ? a[j].z : a[j].w;
                    const float2 aa = make_float2(av, av);
#pragma unroll
                    for (int i = 0; i < NP2; ++i)
                        acc[j][i] = __ffma2_rn(aa, make_float2(w[2 * i], w[2 * i + 1]), acc[j][i]);
                }
            }
        }
    }
    if constexpr (INPLACE) group_sync<T>(group);
    const bool full = g * NI + NI <= N;  // all NI outputs of this thread exist
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        const int row = (qg + QG * j) * OS;
        float v[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            v[i] = NI == 1 ? acc1[j] : ((i & 1) ? acc[j][i >> 1].y : acc[j][i >> 1].x);
            if (mode == 1) v[i] = fmaxf(v[i], 0.0f);
        }
        if constexpr (NI % 4 == 0) {
            if (full) {
#pragma unroll
                for (int i = 0; i < NI; i += 4)
                    *reinterpret_cast<float4*>(out + row + g * NI + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                continue;
            }
        }
#pragma unroll
        for (int i = 0; i < NI; ++i)
            if (g * NI + i < N) out[row + g * NI + i] = v[i];
    }
}

// One layer for the tile; only the register tiles up to NIMAX outputs per
// thread are instantiated (NP = 16 NI <= 16 * NIMAX is guaranteed by the
// launcher). AST as in tile_gemm.
template <int NIMAX, int AST = 0, bool INPLACE = false, int WPAD = 0, int T = kNT>
__device__ __forceinline__ void layer(int t, const float* in, int AS, int K, const float* WT, int NP,
                                      float* out, int OS, int N, int mode, int group = 0) {
    if (NP == 16) tile_gemm<1, AST, INPLACE, WPAD, T>(t, in, AS, K, WT, out, OS, N, mode, group);
    else if (NIMAX >= 2 && NP == 32)
        tile_gemm<(NIMAX >= 2 ? 2 : 1), AST, INPLACE, WPAD, T>(t, in, AS, K, WT, out, OS, N, mode, group);
    else if (NIMAX >= 4 && NP == 64)
        tile_gemm<(NIMAX >= 4 ? 4 : 1), AST, INPLACE, WPAD, T>(t, in, AS, K, WT, out, OS, N, mode, group);
    else if (NIMAX >= 8)
        tile_gemm<(NIMAX >= 8 ? 8 : 1), AST, INPLACE, WPAD, T>(t, in, AS, K, WT, out, OS, N, mode, group);
}

// ------------------------------------------------------------- encode

// Blend of level l at cell cl (F features) into s[0..F).
__device__ __forceinline__ void gather_level(const DevCfg& cfg, const float* __restrict__ grid, int l,
                                             const Cell& cl, float (&s)[8]) {
    const int F = cfg.feat;
    const float* gl = grid + (size_t)cfg.level_off[l] * F;
    uint32_t idx[8];
    corner_idx8(cfg, l, cl, idx);
    float w[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) s[f] = 0.0f;
    if (F == 2) {
        float2 v[8];
#pragma unroll
        for (int c = 0; c < 8; c += 2) gather_pair2(gl, cfg.level_off[l] + cfg.grid_shift, idx[c], idx[c + 1], v[c], v[c + 1]);
        corner_w8(cl, w);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            s[0] = fmaf(w[c], v[c].x, s[0]);
            s[1] = fmaf(w[c], v[c].y, s[1]);
        }
    } else if (F == 4) {
        float4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = __ldg(reinterpret_cast<const float4*>(gl) + idx[c]);
        corner_w8(cl, w);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            s[0] = fmaf(w[c], v[c].x, s[0]);
            s[1] = fmaf(w[c], v[c].y, s[1]);
            s[2] = fmaf(w[c], v[c].z, s[2]);
            s[3] = fmaf(w[c], v[c].w, s[3]);
        }
    } else {
        corner_w8(cl, w);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float* e = gl + (size_t)idx[c] * F;
#pragma unroll
            for (int f = 0; f < 8; ++f)
                if (f < F) s[f] = fmaf(w[c], __ldg(e + f), s[f]);
        }
    }
}

// Fills act[q][0 .. widths[0]) for the tile's 64 queries; local thread t of T
// handles query t % 64 and every (T / 64)-th level (two levels in flight).
// FOUR: 2-feature grids keep four levels' loads in flight (registers the
// wide instances have to spare).
template <bool FOUR, int T = kNT>
__device__ __forceinline__ void encode_tile(int t, const DevCfg& cfg, const float* __restrict__ grid,
                                            int64_t base, int64_t n, int64_t ld,
                                            const float* __restrict__ pos,
                                            const float* __restrict__ aux, float* act, int AS) {
    constexpr int P = T / kTQ;  // threads of a query
    const int q = t & (kTQ - 1), part = t >> 6;
    const int64_t j = base + q;
    const bool valid = j < n;
    float x = 0.0f, y = 0.0f, z = 0.0f;
    if (valid) {
        x = pos[j];
        y = pos[ld + j];
        z = pos[2 * ld + j];
    }
    float* row = act + q * AS;
    const int F = cfg.feat;
    int l = part;
    if (FOUR && F == 2) {
        // Four levels' corner loads in flight (levels l, l + P, ...).
        for (; l + 3 * P < cfg.n_levels; l += 4 * P) {
            Cell cs[4];
            uint32_t idx[4][8];
            float2 v[4][8];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                cs[r] = make_cell(x, y, z, cfg.level_res[l + P * r]);
                corner_idx8(cfg, l + P * r, cs[r], idx[r]);
                const float* gr = grid + (size_t)cfg.level_off[l + P * r] * 2;
#pragma unroll
                for (int c = 0; c < 8; c += 2)
                    gather_pair2(gr, cfg.level_off[l + P * r] + cfg.grid_shift, idx[r][c], idx[r][c + 1], v[r][c], v[r][c + 1]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float w[8];
                corner_w8(cs[r], w);
                float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    a0 = fmaf(w[c], v[r][c].x, a0);
                    a1 = fmaf(w[c], v[r][c].y, a1);
                }
                row[(l + P * r) * 2] = a0;
                row[(l + P * r) * 2 + 1] = a1;
            }
        }
    }
    for (; l + P < cfg.n_levels; l += 2 * P) {
        const Cell c0 = make_cell(x, y, z, cfg.level_res[l]);
        const Cell c1 = make_cell(x, y, z, cfg.level_res[l + P]);
        float s0[8], s1[8];
        gather_level(cfg, grid, l, c0, s0);
        gather_level(cfg, grid, l + P, c1, s1);
#pragma unroll
        for (int f = 0; f < 8; ++f)
            if (f < F) {
                row[l * F + f] = s0[f];
                row[(l + P) * F + f] = s1[f];
            }
    }
    for (; l < cfg.n_levels; l += P) {
        const Cell c0 = make_cell(x, y, z, cfg.level_res[l]);
        float s0[8];
        gather_level(cfg, grid, l, c0, s0);
#pragma unroll
        for (int f = 0; f < 8; ++f)
            if (f < F) row[l * F + f] = s0[f];
    }
    const int o = cfg.grid_feats;
    const int w0 = cfg.widths[0];
    if (cfg.mode == NPM_PRODUCT) {
        if (part == 0) {
            float wo[3] = {0.0f, 0.0f, 1.0f};
            if (valid) {
                wo[0] = aux[j];
                wo[1] = aux[ld + j];
                wo[2] = aux[2 * ld + j];
            }
            float sh[16];
            sh_band4(wo[0], wo[1], wo[2], sh);
#pragma unroll
            for (int i = 0; i < 16; ++i) row[o + i] = sh[i];
        } else if (part == 1) {
            float nn[3] = {0.0f, 0.0f, 1.0f}, r = 0.0f;
            if (valid) {
                nn[0] = aux[3 * ld + j];
                nn[1] = aux[4 * ld + j];
                nn[2] = aux[5 * ld + j];
                r = aux[6 * ld + j];
            }
            float sh[4];
            sh_band2(nn[0], nn[1], nn[2], sh);
#pragma unroll
            for (int i = 0; i < 4; ++i) row[o + 16 + i] = sh[i];
            row[o + 20] = r;
            for (int i = o + 21; i < w0; ++i) row[i] = 0.0f;
        }
    } else if (part == 1) {
        for (int i = o; i < w0; ++i) row[i] = 0.0f;
    }
}

// -------------------------------------------------------- vMF epilogue

// Mapping of one half of the lobes of query q (Table 1). Returns the local
// lobe count; lam holds normalised weights.
template <int KH>
struct HalfMix {
    Lobe lob[KH];
    float cn[KH];
    float mx, ssum;  // largest weight logit and sum of e^{logit - mx}, both halves
    int l0, cnt;
};

template <int KH>
__device__ __forceinline__ void decode_half(const DevCfg& cfg, const float* raw, int half,
                                            HalfMix<KH>& hm, float* mix_out, int64_t ld, int64_t j,
                                            bool valid) {
    const int K = cfg.K, kh = (K + 1) >> 1;
    hm.l0 = half * kh;
    hm.cnt = min(K, hm.l0 + kh) - hm.l0;
    float mx = -INFINITY;
#pragma unroll
    for (int ii = 0; ii < KH; ++ii)
        if (ii < hm.cnt) mx = fmaxf(mx, raw[4 * (hm.l0 + ii)]);
    mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 1));
    float ssum = 0.0f;
#pragma unroll
    for (int ii = 0; ii < KH; ++ii)
        if (ii < hm.cnt) {
            hm.lob[ii].lam = __expf(raw[4 * (hm.l0 + ii)] - mx);
            ssum += hm.lob[ii].lam;
        }
    ssum += __shfl_xor_sync(kFull, ssum, 1);
    hm.mx = mx;
    hm.ssum = ssum;
    const float inv = __fdividef(1.0f, ssum);  // ssum in [1, K]
#pragma unroll
    for (int ii = 0; ii < KH; ++ii)
        if (ii < hm.cnt) {
            const int i = hm.l0 + ii;
            hm.lob[ii].lam *= inv;
            float th, ph;
            decode_lobe_fast(cfg.kappa_act, raw[4 * i + 1], raw[4 * i + 2], raw[4 * i + 3], hm.lob[ii],
                        &th, &ph);
            hm.cn[ii] = vmf_scaled_norm_fast(hm.lob[ii].kap);
            if (mix_out && valid) {
                mix_out[(4 * i + 0) * ld + j] = hm.lob[ii].lam;
                mix_out[(4 * i + 1) * ld + j] = hm.lob[ii].kap;
                mix_out[(4 * i + 2) * ld + j] = th;
                mix_out[(4 * i + 3) * ld + j] = ph;
            }
        }
}

template <int KH>
__device__ __forceinline__ float half_pdf(const HalfMix<KH>& hm, const float w[3]) {
    float pv = 0.0f;
#pragma unroll
    for (int ii = 0; ii < KH; ++ii)
        if (ii < hm.cnt) pv += hm.lob[ii].lam * vmf_eval_fast(hm.lob[ii], hm.cn[ii], w[0], w[1], w[2]);
    return pv + __shfl_xor_sync(kFull, pv, 1);
}

// log V at w (Eq. 4 in log-sum-exp form): the log of each lobe's term,
// log lambda_i + log c(kappa_i) + kappa_i (mu_i.w - 1), with log lambda_i
// taken from the logits so that it stays finite where lambda_i underflows.
template <int KH>
__device__ __forceinline__ float half_log_pdf(const HalfMix<KH>& hm, const float* raw, const float w[3]) {
    const float lnorm = hm.mx + __logf(hm.ssum);
    float a[KH];
    float m = -INFINITY;
#pragma unroll
    for (int ii = 0; ii < KH; ++ii)
        if (ii < hm.cnt) {
            const Lobe& L = hm.lob[ii];
            const float d = L.mu[0] * w[0] + L.mu[1] * w[1] + L.mu[2] * w[2];
            a[ii] = (raw[4 * (hm.l0 + ii)] - lnorm) + __logf(hm.cn[ii]) + L.kap * (d - 1.0f);
            m = fmaxf(m, a[ii]);
        }
    m = fmaxf(m, __shfl_xor_sync(kFull, m, 1));
    float s = 0.0f;
#pragma unroll
    for (int ii = 0; ii < KH; ++ii)
        if (ii < hm.cnt) s += __expf(a[ii] - m);
    s += __shfl_xor_sync(kFull, s, 1);
    return m + __logf(s);
}

template <bool SAMPLE, int KH>
__device__ __forceinline__ void epilogue_tile(int t, const DevCfg& cfg, const float* act, int AS,
                                              int64_t base, int64_t n, int64_t ld,
                                              const float* __restrict__ uin, float ufrac,
                                              float* __restrict__ dir_out,
                                              float* __restrict__ pdf_out,
                                              float* __restrict__ mix_out, bool log_pdf = false) {
    const int q = t >> 1, half = t & 1;
    const int64_t j = base + q;
    const bool valid = j < n;
    const float* raw = act + q * AS;
    HalfMix<KH> hm;
    decode_half(cfg, raw, half, hm, mix_out, ld, j, valid);
    float w[3];
    bool uni = false;
    if (SAMPLE) {
        float u0 = 0.0f, u1 = 0.0f, u2 = 0.0f;
        if (valid) {
            u0 = uin[j];
            u1 = uin[ld + j];
            u2 = uin[2 * ld + j];
            uni = ufrac > 0.0f && uin[3 * ld + j] < ufrac;
        }
        // Lobe choice: smallest i with u0 < lambda_0 + ... + lambda_i, the
        // cumulative sum taken in lobe order: half 0 sums its lobes from 0,
        // half 1 continues from half 0's total.
        float run = 0.0f;
        int sel = -1;
        if (half == 0) {
#pragma unroll
            for (int ii = 0; ii < KH; ++ii)
                if (ii < hm.cnt) {
                    run += hm.lob[ii].lam;
                    if (sel < 0 && u0 < run) sel = ii;
                }
        }
        const float tot0 = __shfl_xor_sync(kFull, run, 1);
        if (half == 1) {
            float cum = tot0;
#pragma unroll
            for (int ii = 0; ii < KH; ++ii)
                if (ii < hm.cnt) {
                    cum += hm.lob[ii].lam;
                    if (sel < 0 && u0 < cum) sel = ii;
                }
        }
        const int osel = __shfl_xor_sync(kFull, sel, 1);
        const int sel0 = half ? osel : sel, sel1 = half ? sel : osel;
        const int kh = (cfg.K + 1) >> 1;
        int owner, lidx;
        if (sel0 >= 0) {
            owner = 0;
            lidx = sel0;
        } else if (sel1 >= 0) {
            owner = 1;
            lidx = sel1;
        } else {
            const int last = cfg.K - 1;
            owner = last >= kh ? 1 : 0;
            lidx = last - owner * kh;
        }
        float d[3] = {0.0f, 0.0f, 1.0f};
        if (half == owner) {
            if (uni) {
                uniform_sphere(u1, u2, d);
            } else {
                Lobe sl = hm.lob[0];
#pragma unroll
                for (int ii = 1; ii < KH; ++ii)
                    if (ii == lidx) sl = hm.lob[ii];
                vmf_sample(sl, u1, u2, d);
            }
        }
        const int src = (threadIdx.x & 31 & ~1) | owner;
#pragma unroll
        for (int a = 0; a < 3; ++a) w[a] = __shfl_sync(kFull, d[a], src);
    } else {
        w[0] = w[1] = 0.0f;
        w[2] = 1.0f;
        if (valid) {
            w[0] = uin[j];
            w[1] = uin[ld + j];
            w[2] = uin[2 * ld + j];
        }
    }
    float pv;
    if (!SAMPLE && log_pdf) {
        pv = half_log_pdf(hm, raw, w);
    } else {
        pv = half_pdf(hm, w);
        if (SAMPLE && ufrac > 0.0f) pv = ufrac * kInv4Pi + (1.0f - ufrac) * pv;
    }
    if (valid) {
        if (half == 0) {
            if (SAMPLE) {
                dir_out[j] = w[0];
                dir_out[ld + j] = w[1];
                dir_out[2 * ld + j] = w[2];
            }
        } else {
            pdf_out[j] = pv;
        }
    }
}

// ------------------------------------------------------ forward kernel

// One CTA per SM holds G tile groups of 128 threads. The groups share one
// copy of the weights in shared memory and each walks its own 64-query tiles
// with its own activation buffers and named barrier.
template <bool SAMPLE, int NIMAX, int KH>
__global__ void __launch_bounds__(fwd_max_groups(NIMAX) * kNT, 1) k_forward_fp32(const __grid_constant__ DevCfg cfg,
                                                         const float* __restrict__ grid,
                                                         const float* __restrict__ wfwd,
                                                         const __grid_constant__ QueryBatch qb) {
    extern __shared__ float4 smem4[];
    float* sW = reinterpret_cast<float*>(smem4);
    constexpr int AS = fwd_act_stride(NIMAX);
    const int G = blockDim.x / kNT;
    const int group = threadIdx.x / kNT;
    const int t = threadIdx.x % kNT;
    float* act = sW + cfg.fwd_floats + group * kTQ * AS;  // one tile, layers in place
    for (int i = threadIdx.x; i < cfg.fwd_floats / 4; i += blockDim.x)
        smem4[i] = __ldg(reinterpret_cast<const float4*>(wfwd) + i);
    __syncthreads();
    int64_t total = qb.total_tiles, n0 = qb.seg[0].n;
    if (qb.n_dev) {
        n0 = *qb.n_dev;
        total = (n0 + kTQ - 1) / kTQ;
    }
    for (int64_t tile = (int64_t)blockIdx.x * G + group; tile < total; tile += (int64_t)gridDim.x * G) {
        int s = 0;
        while (s + 1 < qb.nseg && tile >= qb.seg[s + 1].tile0) ++s;
        const QuerySeg& S = qb.seg[s];
        const int64_t n = (s == 0 && qb.n_dev) ? n0 : S.n;
        const int64_t base = (tile - S.tile0) * kTQ;
        encode_tile<(NIMAX >= 4)>(t, cfg, grid, base, n, S.ld, S.pos, S.aux, act, AS);
        group_sync(group);
        // Bring the next tile's positions and this tile's uniforms into L2
        // while the MLP runs (one thread per 32 consecutive queries).
        if ((t & 31) == 0 && t < 2 * kTQ) {
            const int row = t >> 5;  // 0..3: u rows 0..2 of this tile, pos of the next
            if (row < 3) {
                const int64_t jj = base + (t & (kTQ - 1));
                if (jj < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(S.uin + row * S.ld + jj));
            } else {
                const int64_t nt = tile + (int64_t)gridDim.x * G;
                if (nt < total) {
                    int s2 = s;
                    while (s2 + 1 < qb.nseg && nt >= qb.seg[s2 + 1].tile0) ++s2;
                    const QuerySeg& S2 = qb.seg[s2];
                    const int64_t b2 = (nt - S2.tile0) * kTQ;
                    for (int r = 0; r < 3; ++r) {
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(S2.pos + r * S2.ld + b2));
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(S2.pos + r * S2.ld + b2 + 32));
                    }
                }
            }
        }
        for (int l = 0; l < cfg.n_layers; ++l) {
            const bool last = l == cfg.n_layers - 1;
            layer<NIMAX, AS, true>(t, act, AS, cfg.widths[l], sW + cfg.off_fwd[l], cfg.np_fwd[l], act, AS,
                                   cfg.widths[l + 1], last ? 0 : 1, group);
            group_sync(group);
        }
        epilogue_tile<SAMPLE, KH>(t, cfg, act, AS, base, n, S.ld, S.uin, S.ufrac, S.dir, S.pdf, S.mix,
                                      qb.log_pdf != 0);
        group_sync(group);
    }
}

// ------------------------------------------------------ training kernel

// Threads of a training tile group: four per query of its 64-query tiles.
constexpr int kTrainT = 256;

// Per query: raw outputs -> d(sum_j s_j log V_j)/d raw, written in place,
// and s_j log V_j added to lacc. Log-domain mixture so that log V
// and the responsibilities r_i stay finite when V underflows FP32.
template <int P>
__device__ __forceinline__ void grad_epilogue(int t, const DevCfg& cfg, float* act, int AS, int64_t base,
                                              int64_t n, int64_t ld,
                                              const float* __restrict__ dir,
                                              const float* __restrict__ rad,
                                              const float* __restrict__ spdf,
                                              const float* __restrict__ dlogv, float inv_n, float& lacc) {
    const int q = t / P, part = t % P;
    const int64_t j = base + q;
    const bool valid = j < n;
    float* raw = act + q * AS;
    const int K = cfg.K, KH = (K + P - 1) / P;
    const int l0 = part * KH, cnt = min(K, l0 + KH) - l0;  // (none where the others hold all)
    float w[3] = {0.0f, 0.0f, 1.0f};
    float s = 0.0f;
    if (valid) {
        w[0] = dir[j];
        w[1] = dir[ld + j];
        w[2] = dir[2 * ld + j];
        s = dlogv ? dlogv[j] : -(rad[j] / spdf[j]) * inv_n;
    }
    constexpr int H = NPM_MAX_LOBES / P;
    float lp[H], a[H], kap[H], md[H], wdt[H], wdp[H], sk[H], st[H], sp[H];
    float mx = -INFINITY;
#pragma unroll
    for (int ii = 0; ii < H; ++ii)
        if (ii < cnt) mx = fmaxf(mx, raw[4 * (l0 + ii)]);
#pragma unroll
    for (int o = 1; o < P; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    float ssum = 0.0f;
#pragma unroll
    for (int ii = 0; ii < H; ++ii)
        if (ii < cnt) ssum += expf(raw[4 * (l0 + ii)] - mx);
#pragma unroll
    for (int o = 1; o < P; o <<= 1) ssum += __shfl_xor_sync(kFull, ssum, o);
    const float lse = mx + logf(ssum);
    float amax = -INFINITY;
#pragma unroll
    for (int ii = 0; ii < H; ++ii)
        if (ii < cnt) {
            const int i = l0 + ii;
            lp[ii] = raw[4 * i] - lse;  // log lambda_i
            const float rk = raw[4 * i + 1];
            if (cfg.kappa_act == NPM_EXP) {
                kap[ii] = expf(rk);
                sk[ii] = kap[ii];
            } else {
                kap[ii] = softplus(rk);
                sk[ii] = logistic(rk);
            }
            st[ii] = logistic(raw[4 * i + 2]);
            sp[ii] = logistic(raw[4 * i + 3]);
            float sth, cth, sph, cph;
            sincosf(kPi * st[ii], &sth, &cth);
            sincosf(2.0f * kPi * sp[ii], &sph, &cph);
            md[ii] = sth * cph * w[0] + sth * sph * w[1] + cth * w[2];
            wdt[ii] = cth * cph * w[0] + cth * sph * w[1] - sth * w[2];
            wdp[ii] = -sth * sph * w[0] + sth * cph * w[1];
            a[ii] = lp[ii] + logf(vmf_scaled_norm(kap[ii])) + kap[ii] * (md[ii] - 1.0f);
            amax = fmaxf(amax, a[ii]);
        }
#pragma unroll
    for (int o = 1; o < P; o <<= 1) amax = fmaxf(amax, __shfl_xor_sync(kFull, amax, o));
    float es = 0.0f;
#pragma unroll
    for (int ii = 0; ii < H; ++ii)
        if (ii < cnt) es += expf(a[ii] - amax);
#pragma unroll
    for (int o = 1; o < P; o <<= 1) es += __shfl_xor_sync(kFull, es, o);
    const float logV = amax + logf(es);
#pragma unroll
    for (int ii = 0; ii < H; ++ii)
        if (ii < cnt) {
            const int i = l0 + ii;
            const float r = expf(a[ii] - logV);
            const float lam = expf(lp[ii]);
            const float sr = s * r;
            raw[4 * i + 0] = s * (r - lam);
            raw[4 * i + 1] = sr * (inv_minus_coth(kap[ii]) + md[ii]) * sk[ii];
            raw[4 * i + 2] = sr * kap[ii] * wdt[ii] * kPi * st[ii] * (1.0f - st[ii]);
            raw[4 * i + 3] = sr * kap[ii] * wdp[ii] * 2.0f * kPi * sp[ii] * (1.0f - sp[ii]);
        }
    if (valid && part == 0) lacc += s * logV;
}

// dW[n][k] += sum_q dl[q][n] * h[q][k] (global atomics); row strides DS, HS.
// Thread t of 256 owns 4 x 4 blocks.
__device__ __forceinline__ void weight_grad(int t, const float* dl, int DS, const float* h, int HS, int N, int K,
                                            float* __restrict__ gW) {
    const bool wide = (reinterpret_cast<uintptr_t>(gW) & 15u) == 0;
    for (int n0 = (t >> 4) * 4; n0 < N; n0 += 64)
        for (int k0 = (t & 15) * 4; k0 < K; k0 += 64) {
            float2 acc[4][2];
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = make_float2(0.0f, 0.0f);
#pragma unroll 4
            for (int q = 0; q < kTQ; ++q) {
                const float4 hv = *reinterpret_cast<const float4*>(h + q * HS + k0);
                const float4 d = *reinterpret_cast<const float4*>(dl + q * DS + n0);
                const float2 h0 = make_float2(hv.x, hv.y), h1 = make_float2(hv.z, hv.w);
                const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float2 dd = make_float2(dv[r], dv[r]);
                    acc[r][0] = __ffma2_rn(dd, h0, acc[r][0]);
                    acc[r][1] = __ffma2_rn(dd, h1, acc[r][1]);
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                // (8-byte aligned: the gradient shares the tables' shift)
                red_add4(gW + (size_t)(n0 + r) * K + k0, wide, acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
            }
        }
}

// The layer's input gradient in place of its input h: h[q][k] =
// (sum_n dl[q][n] W[n][k]) where h[q][k] > 0 (ReLU's derivative; everywhere
// without relu), from the forward pass's copy of the weights, W^T rows of WS
// floats. Thread (qg, g) of 256 owns queries qg + 16 j and inputs g + 16 i; the sums
// run over n in packed pairs. WS = np + 4 keeps the 16 rows that a warp reads
// at once on different banks.
__device__ __forceinline__ void input_grad(int t, const float* dl, int DS, int N, const float* __restrict__ WT, int WS,
                                           float* h, int HS, int K, bool relu) {
    constexpr int KI = 4, NQ = 4;  // inputs a thread and pass, queries
    const int g = (t & 31) >> 1, qg = (t & 1) | ((t >> 5) << 1);
    for (int k0 = 0; k0 < K; k0 += 16 * KI) {
        float2 acc[NQ][KI];
#pragma unroll
        for (int j = 0; j < NQ; ++j)
#pragma unroll
            for (int i = 0; i < KI; ++i) acc[j][i] = make_float2(0.0f, 0.0f);
        // Rows past K repeat the last one (their sums are not stored).
        const float* wr[KI];
#pragma unroll
        for (int i = 0; i < KI; ++i) wr[i] = WT + min(k0 + g + 16 * i, K - 1) * WS;
        for (int n = 0; n < N; n += 4) {
            float4 w[KI];
#pragma unroll
            for (int i = 0; i < KI; ++i) w[i] = *reinterpret_cast<const float4*>(wr[i] + n);
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const float4 a = *reinterpret_cast<const float4*>(dl + (qg + 16 * j) * DS + n);
                const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
#pragma unroll
                for (int i = 0; i < KI; ++i) {
                    acc[j][i] = __ffma2_rn(a0, make_float2(w[i].x, w[i].y), acc[j][i]);
                    acc[j][i] = __ffma2_rn(a1, make_float2(w[i].z, w[i].w), acc[j][i]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < NQ; ++j)
#pragma unroll
            for (int i = 0; i < KI; ++i) {
                const int k = k0 + g + 16 * i;
                if (k < K) {
                    float* o = h + (qg + 16 * j) * HS + k;
                    *o = !relu || *o > 0.0f ? acc[j][i].x + acc[j][i].y : 0.0f;
                }
            }
    }
}

// Grid gradient: dV_l[corner] += weight * dG_l (Eq. 11 transposed).
__device__ __forceinline__ void grid_scatter(int t, const DevCfg& cfg, const float* denc, int AS,
                                             int64_t base, int64_t n, int64_t ld,
                                             const float* __restrict__ pos,
                                             float* __restrict__ ggrid) {
    const int q = t & (kTQ - 1), part = t >> 6;
    const int64_t j = base + q;
    if (j >= n) return;
    const float x = pos[j], y = pos[ld + j], z = pos[2 * ld + j];
    const float* row = denc + q * AS;
    const int F = cfg.feat;
    for (int l = part; l < cfg.n_levels; l += kTrainT / kTQ) {
        const Cell cl = make_cell(x, y, z, cfg.level_res[l]);
        float* gl = ggrid + (size_t)cfg.level_off[l] * F;
        const float* dg = row + l * F;
        uint32_t idx[8];
        float ws[8];
        corners8(cfg, l, cl, idx, ws);
        if (F == 2) {
#pragma unroll
            for (int c = 0; c < 8; c += 2)
                scatter_pair2(gl, cfg.level_off[l] + cfg.grid_shift, idx[c], idx[c + 1], ws[c], ws[c + 1], dg[0], dg[1]);
            continue;
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float w = ws[c];
            float* e = gl + (size_t)idx[c] * F;
            if (F == 4) {
                red_add(e, w * dg[0], w * dg[1], w * dg[2], w * dg[3]);
            } else {
                for (int f = 0; f < F; ++f) red_add(e + f, w * dg[f]);
            }
        }
    }
}

// Floats of a CTA's shared memory: the weights, W^T rows padded by 4, and per
// tile group the input and every layer's output of a 64-query tile, rows
// padded by 4.
constexpr int kPad = 4;
__host__ __device__ inline int train_weight_floats(const DevCfg& c) {
    int n = 0;
    for (int l = 0; l < c.n_layers; ++l) n += c.widths[l] * (c.np_fwd[l] + kPad);
    return n;
}
__host__ __device__ inline int train_group_floats(const DevCfg& c) {
    int n = 0;
    for (int l = 0; l <= c.n_layers; ++l) n += kTQ * (c.widths[l] + kPad);
    return n;
}

// Tile groups of 256 threads share the weights; each walks its own 64-query
// tiles. A layer's gradient replaces its activations in place, and forward
// and backward read one copy of the weights, so two groups (16 warps) fit
// beside it on the 64-wide networks. Bound by FMA issue and shared-memory
// operands, which share the L1 data pipe. Against one group of 128 threads
// with one buffer more and the backward weights in global memory (GB300):
// 65,551 samples of the eight-level grid into 64-wide layers 370 -> 214 us,
// 20,011 of the product-mode network 200 -> 135 us (two groups of 128
// threads: 301 against 261 us for the whole step of the first).
constexpr int kTrainGroups = 2;

__global__ void __launch_bounds__(kTrainGroups* kTrainT, 1)
    k_train_fp32(const __grid_constant__ DevCfg cfg, const float* __restrict__ params, int64_t mlp_off,
                 const float* __restrict__ wfwd, int64_t n, int64_t ld, const float* __restrict__ pos,
                 const float* __restrict__ aux, const float* __restrict__ dir, const float* __restrict__ rad,
                 const float* __restrict__ spdf, const float* __restrict__ dlogv, float inv_n,
                 float* __restrict__ grad, double* __restrict__ loss) {
    extern __shared__ float4 smem4[];
    grid_dep_launch();
    float* sW = reinterpret_cast<float*>(smem4);
    const int L = cfg.n_layers;
    const int G = blockDim.x / kTrainT, group = threadIdx.x / kTrainT, t = threadIdx.x % kTrainT;
    float* buf0 = sW + train_weight_floats(cfg) + group * train_group_floats(cfg);
    {
        int o = 0;
        for (int l = 0; l < L; ++l) {
            const int np4 = cfg.np_fwd[l] / 4, ws4 = (cfg.np_fwd[l] + kPad) / 4;
            const float4* src = reinterpret_cast<const float4*>(wfwd + cfg.off_fwd[l]);
            for (int i = threadIdx.x; i < cfg.widths[l] * np4; i += blockDim.x)
                smem4[o + i / np4 * ws4 + i % np4] = __ldg(src + i);
            o += cfg.widths[l] * ws4;
        }
    }
    __syncthreads();
    float lacc = 0.0f;  // this thread's share of the loss
    const int64_t ntiles = (n + kTQ - 1) / kTQ;
    for (int64_t tile = blockIdx.x + (int64_t)group * gridDim.x; tile < ntiles; tile += (int64_t)gridDim.x * G) {
        const int64_t base = tile * kTQ;
        float* buf = buf0;
        const float* w = sW;
        encode_tile<false, kTrainT>(t, cfg, params, base, n, ld, pos, aux, buf, cfg.widths[0] + kPad);
        group_sync<kTrainT>(group);
        for (int l = 0; l < L; ++l) {
            const int IS = cfg.widths[l] + kPad, OS = cfg.widths[l + 1] + kPad;
            float* out = buf + kTQ * IS;
            layer<8, 0, false, kPad, kTrainT>(t, buf, IS, cfg.widths[l], w, cfg.np_fwd[l], out, OS, cfg.widths[l + 1],
                                     l == L - 1 ? 0 : 1, group);
            group_sync<kTrainT>(group);
            buf = out;
            w += cfg.widths[l] * (cfg.np_fwd[l] + kPad);
        }
        grad_epilogue<kTrainT / kTQ>(t, cfg, buf, cfg.widths[L] + kPad, base, n, ld, dir, rad, spdf, dlogv, inv_n, lacc);
        group_sync<kTrainT>(group);
        // Backward: the gradient of layer l's output lies in buf; that of its
        // input takes the place of the input.
        float* gW = grad + mlp_off;
        for (int l = 0; l < L; ++l) gW += cfg.widths[l] * cfg.widths[l + 1];
        for (int l = L - 1; l >= 0; --l) {
            const int N = cfg.widths[l + 1], K = cfg.widths[l];
            float* h = buf - kTQ * (K + kPad);
            w -= K * (cfg.np_fwd[l] + kPad);
            gW -= K * N;
            weight_grad(t, buf, N + kPad, h, K + kPad, N, K, gW);
            group_sync<kTrainT>(group);
            input_grad(t, buf, N + kPad, N, w, cfg.np_fwd[l] + kPad, h, K + kPad, K, l > 0);
            group_sync<kTrainT>(group);
            buf = h;
        }
        grid_scatter(t, cfg, buf, cfg.widths[0] + kPad, base, n, ld, pos, grad);
        group_sync<kTrainT>(group);
    }
    // The loss: one atomic a warp.
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lacc += __shfl_xor_sync(kFull, lacc, o);
    if (loss && (t & 31) == 0 && lacc != 0.0f) atomicAdd(loss, (double)lacc);
}

// ------------------------------------------------------- utility kernels

// blockIdx.y: layer.
__global__ void k_arrange_weights(const __grid_constant__ DevCfg cfg, const float* mlp, float* __restrict__ wfwd,
                                  UpdateEnd end) {
    grid_dep_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) end_update(end);
    arrange_layer(cfg, blockIdx.y, mlp, wfwd, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// Dense Adam with bias correction (Kingma and Ba) at step t = *steps + 1,
// c1 = 1 - b1^t, c2 = 1 - b2^t; the step count lives in device memory so that
// captured graphs replay correctly (end_update advances it afterwards).
// Skips the update when *loss is not finite and flags it. Clears the
// gradient. Optionally refreshes an FP16 copy of the first n_half parameters
// (the grid). With ema set, also the exponential moving average
// e <- d e + (1 - d) p of the updated parameters that inference evaluates
// (Sec. 5.3); the FP16 copy (inference only) is then taken from e.
__global__ void k_adam(int64_t n4, float4* p, float4* g, float4* m, float4* v, float lr, float b1, float b2,
                       float eps, const int* steps, const double* loss, int* __restrict__ status,
                       __half2* __restrict__ half_copy, int64_t n_half, float4* ema, float ema_decay) {
    grid_dep_wait();
    grid_dep_launch();
    const bool skip = loss != nullptr && !isfinite((float)*loss);
    if (skip && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, kStatusNumeric);
    const float t = (float)(*steps + 1);
    const float c1 = 1.0f - powf(b1, t), c2 = 1.0f - powf(b2, t);
    // Two float4 groups per thread and iteration: more bytes in flight.
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < n4; i0 += 2 * stride) {
        float4 gg[2], mm[2], vv[2], pp[2];
        bool in[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t i = i0 + u * stride;
            in[u] = i < n4;
            if (in[u]) {
                gg[u] = g[i];
                mm[u] = m[i];
                vv[u] = v[i];
                pp[u] = p[i];
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t i = i0 + u * stride;
            if (!in[u]) continue;
            g[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (skip) continue;
            float* pm = &mm[u].x;
            float* pv = &vv[u].x;
            const float* pg = &gg[u].x;
            float* pq = &pp[u].x;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                pm[c] = b1 * pm[c] + (1.0f - b1) * pg[c];
                pv[c] = b2 * pv[c] + (1.0f - b2) * pg[c] * pg[c];
                const float mh = pm[c] / c1, vh = pv[c] / c2;
                pq[c] -= lr * mh / (sqrtf(vh) + eps);
            }
            m[i] = mm[u];
            v[i] = vv[u];
            p[i] = pp[u];
            float4 inf = pp[u];
            if (ema) {
                float4 e = ema[i];
                const float d = ema_decay, d1 = 1.0f - ema_decay;
                e.x = d * e.x + d1 * pp[u].x;
                e.y = d * e.y + d1 * pp[u].y;
                e.z = d * e.z + d1 * pp[u].z;
                e.w = d * e.w + d1 * pp[u].w;
                ema[i] = e;
                inf = e;
            }
            if (half_copy && 4 * i < n_half) {
                if (4 * i + 4 <= n_half) {
                    half_copy[2 * i] = __floats2half2_rn(inf.x, inf.y);
                    half_copy[2 * i + 1] = __floats2half2_rn(inf.z, inf.w);
                } else {
                    // The copy's last entries (n_half not a multiple of 4).
                    __half* hc = reinterpret_cast<__half*>(half_copy) + 4 * i;
                    const float iv[4] = {inf.x, inf.y, inf.z, inf.w};
                    for (int c = 0; c < (int)(n_half - 4 * i); ++c) hc[c] = __float2half_rn(iv[c]);
                }
            }
        }
    }
}

__global__ void k_grid_indices(DevCfg cfg, int64_t n, int64_t ld, const float* __restrict__ pos,
                               int32_t* __restrict__ out) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const float x = pos[j], y = pos[ld + j], z = pos[2 * ld + j];
        for (int l = 0; l < cfg.n_levels; ++l) {
            const Cell cl = make_cell(x, y, z, cfg.level_res[l]);
            uint32_t idx[8];
            float w[8];
            corners8(cfg, l, cl, idx, w);  // the routine every encoder and scatter uses
#pragma unroll
            for (int c = 0; c < 8; ++c) out[((int64_t)l * 8 + c) * n + j] = (int32_t)idx[c];
        }
    }
}

// dst0[i] = src0[i] for i < n0 in vectors V, dst1[i] = src1[i] for i < n1: the
// grid and the MLP between the public layout and the library's, in one launch
// at any alignment (a copy call each cost the host two to three times that,
// and ran at half the bandwidth where the two sides' alignments differ).
template <typename V>
__global__ void __launch_bounds__(256) k_copy_params(const V* __restrict__ src0, V* __restrict__ dst0, int64_t n0,
                                                     const float* __restrict__ src1, float* __restrict__ dst1,
                                                     int64_t n1) {
    constexpr int U = 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < n0; i += U * stride) {
        V v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * stride < n0) v[u] = src0[i + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * stride < n0) dst0[i + u * stride] = v[u];
    }
    for (int64_t i = i0; i < n1; i += stride) dst1[i] = src1[i];
}

__global__ void k_to_half(int64_t n, const float* __restrict__ src, __half* __restrict__ dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = __float2half_rn(src[i]);
}

// ----------------------------------------------------------- launchers


// What decides whether a network can be trained in FP32 (part of the
// interface); the kernel's own layout is never larger.
size_t train_smem_bytes(const DevCfg& c) {
    return sizeof(float) *
           ((size_t)c.fwd_floats + (size_t)(c.n_layers + 2) * kTQ * (c.max_width + 4));
}

static int sm_count() {
    static int cached = 0;
    if (!cached) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev);
    }
    return cached;
}

// Shared-memory carveout (percent of the 228 KB maximum) that holds `bytes`.
int carveout_percent(size_t bytes) {
    const size_t max_smem = 228 * 1024;
    int pct = (int)((bytes * 100 + max_smem - 1) / max_smem);
    return pct < 1 ? 1 : pct > 100 ? 100 : pct;
}

// Template instance (register tile of the widest layer, lobes per half).
static int fp32_instance(const DevCfg& cfg) {
    int need = 1;
    for (int l = 0; l < cfg.n_layers; ++l) need = cfg.np_fwd[l] / 16 > need ? cfg.np_fwd[l] / 16 : need;
    // the activation rows (stride fwd_act_stride(I)) hold every width
    const int mw = (cfg.max_width + 15) / 16;
    need = mw > need ? mw : need;
    const int kh = (cfg.K + 1) / 2;
    need = kh > need ? kh : need;
    return need <= 2 ? 2 : need <= 4 ? 4 : 8;
}

// Shared memory of a one-group CTA: weights and one activation tile.
size_t fwd_smem_bytes(const DevCfg& c) {
    return sizeof(float) * ((size_t)c.fwd_floats + (size_t)kTQ * fwd_act_stride(fp32_instance(c)));
}

template <bool SAMPLE, int I>
static cudaError_t launch_fwd_inst(const DevCfg& cfg, const float* grid, const float* wfwd,
                                   const QueryBatch& qb, int64_t tiles_hint, cudaStream_t st) {
    auto kern = k_forward_fp32<SAMPLE, I, I>;
    const size_t wbytes = sizeof(float) * (size_t)cfg.fwd_floats;
    const size_t gbytes = sizeof(float) * (size_t)kTQ * fwd_act_stride(I);
    int G = (int)((227 * 1024 - wbytes) / gbytes);
    if (G > fwd_max_groups(I)) G = fwd_max_groups(I);
    // Tuning override (groups per CTA) for launch-configuration sweeps.
    static std::atomic<int> env_groups{INT32_MIN + 1};
    const int og = env_override("NPM_FP32_GROUPS", env_groups);
    if (og >= 1 && og < G) G = og;
    if (G < 1) return cudaErrorInvalidConfiguration;
    const size_t smem = wbytes + G * gbytes;
    // Carve out only the shared memory this CTA needs; the rest of the
    // 256 KB stays L1 for the grid gathers.
    static std::atomic<uint64_t> attrs{~0ull};
    cudaError_t e = set_smem_attrs(kern, smem, carveout_percent(smem + 1024), attrs);
    if (e != cudaSuccess) return e;
    int64_t g = sm_count();
    const int64_t need = (tiles_hint + G - 1) / G;
    if (need < g) g = need < 1 ? 1 : need;
    kern<<<(int)g, G * kNT, smem, st>>>(cfg, grid, wfwd, qb);
    return cudaGetLastError();
}

cudaError_t launch_forward_fp32_batch(const DevCfg& cfg, const float* grid, const float* wfwd,
                                      QueryBatch& qb, int64_t max_n, cudaStream_t st) {
    int64_t t0 = 0;
    for (int s = 0; s < qb.nseg; ++s) {
        qb.seg[s].tile0 = t0;
        t0 += (qb.seg[s].n + kTQ - 1) / kTQ;
    }
    qb.total_tiles = t0;
    const int64_t hint = qb.n_dev ? (max_n + kTQ - 1) / kTQ : t0;
    const int inst = fp32_instance(cfg);
    // Sampling reaches this path only with weights that the tensor-core
    // forward cannot hold, which takes layers wider than 64.
    if (qb.sample)
        return inst == 8 ? launch_fwd_inst<true, 8>(cfg, grid, wfwd, qb, hint, st) : cudaErrorInvalidConfiguration;
    if (inst == 2) return launch_fwd_inst<false, 2>(cfg, grid, wfwd, qb, hint, st);
    if (inst == 4) return launch_fwd_inst<false, 4>(cfg, grid, wfwd, qb, hint, st);
    return launch_fwd_inst<false, 8>(cfg, grid, wfwd, qb, hint, st);
}

cudaError_t launch_forward_fp32(const DevCfg& cfg, const float* grid, const float* wfwd, int64_t n,
                                int64_t ld, const float* pos, const float* aux, const float* uin,
                                float ufrac, bool sample, float* dir_out, float* pdf_out,
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
    return launch_forward_fp32_batch(cfg, grid, wfwd, qb, n, st);
}

cudaError_t launch_train_fp32(const DevCfg& cfg, const float* params, int64_t mlp_off, const float* wfwd, int64_t n,
                              int64_t ld, const float* pos, const float* aux, const float* dir, const float* rad,
                              const float* spdf, const float* dlogv, float* grad, double* loss, cudaStream_t st) {
    const size_t wbytes = sizeof(float) * train_weight_floats(cfg), gbytes = sizeof(float) * train_group_floats(cfg);
    int G = kTrainGroups;
    while (G > 1 && wbytes + G * gbytes > 227 * 1024) --G;
    const size_t smem = wbytes + G * gbytes;
    static std::atomic<uint64_t> attrs{~0ull};
    cudaError_t e = set_smem_attrs(k_train_fp32, smem, carveout_percent(smem + 1024), attrs);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (n + kTQ - 1) / kTQ;
    int64_t g = sm_count();
    if (ntiles < g) g = ntiles;
    k_train_fp32<<<(int)g, G * kTrainT, smem, st>>>(cfg, params, mlp_off, wfwd, n, ld, pos, aux, dir, rad, spdf, dlogv,
                                                1.0f / (float)n, grad, loss);
    return cudaGetLastError();
}

cudaError_t launch_arrange_weights(const DevCfg& cfg, const float* mlp, float* wfwd, const UpdateEnd& end,
                                   cudaStream_t st) {
    return launch_maybe_pdl(k_arrange_weights, dim3(16, cfg.n_layers), dim3(256), 0, st, true, cfg, mlp, wfwd, end);
}

cudaError_t launch_adam(int64_t n, float* p, float* g, float* m, float* v, float lr, float b1,
                        float b2, float eps, int* steps, const double* loss, int* status,
                        __half* half_copy, int64_t n_half, float* ema, float ema_decay,
                        cudaStream_t st) {
    const int64_t n4 = n / 4;
    int grid = (int)((n4 + 255) / 256);
    const int cap = sm_count() * 16;
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    return launch_maybe_pdl(k_adam, dim3(grid), dim3(256), 0, st, true, n4, reinterpret_cast<float4*>(p),
                            reinterpret_cast<float4*>(g), reinterpret_cast<float4*>(m), reinterpret_cast<float4*>(v),
                            lr, b1, b2, eps, steps, loss, status, reinterpret_cast<__half2*>(half_copy), n_half,
                            reinterpret_cast<float4*>(ema), ema_decay);
}

cudaError_t launch_grid_indices(const DevCfg& cfg, int64_t n, int64_t ld, const float* pos,
                                int32_t* out, cudaStream_t st) {
    int grid = (int)((n + 255) / 256);
    if (grid > 4096) grid = 4096;
    k_grid_indices<<<grid, 256, 0, st>>>(cfg, n, ld, pos, out);
    return cudaGetLastError();
}

cudaError_t launch_copy_params(const float* src0, float* dst0, int64_t n0, const float* src1, float* dst1, int64_t n1,
                               cudaStream_t st) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src0) | reinterpret_cast<uintptr_t>(dst0) |
                        (uintptr_t)(n0 * (int64_t)sizeof(float));
    const int64_t cap = (int64_t)sm_count() * 8;
    auto launch = [&](auto* v) {
        using V = std::remove_pointer_t<decltype(v)>;
        const int64_t n = n0 * (int64_t)sizeof(float) / (int64_t)sizeof(V);
        int64_t blocks = (n / 4 + n1 / 4 + 255) / 256;
        blocks = blocks < 1 ? 1 : blocks > cap ? cap : blocks;
        k_copy_params<V><<<(int)blocks, 256, 0, st>>>(reinterpret_cast<const V*>(src0), reinterpret_cast<V*>(dst0), n,
                                                      src1, dst1, n1);
    };
    if (a % 16 == 0) launch(static_cast<float4*>(nullptr));
    else if (a % 8 == 0) launch(static_cast<float2*>(nullptr));
    else launch(static_cast<float*>(nullptr));
    return cudaGetLastError();
}

cudaError_t launch_to_half(int64_t n, const float* src, __half* dst, cudaStream_t st) {
    int grid = (int)((n + 255) / 256);
    if (grid > 4096) grid = 4096;
    k_to_half<<<grid, 256, 0, st>>>(n, src, dst);
    return cudaGetLastError();
}

}  // namespace npm
