// npm_tc_forward.cuh -- tensor-core forward pass (encode, MLP, sample and
// density) on sm_103a with the activations in tensor memory.
//
// One persistent CTA per SM holds G tile groups of 128 threads that share one
// copy of the weights in shared memory. Thread t of a group owns query t of
// the group's 128-query tile, which is lane t of its tensor-memory columns.
// Per tile:
//   encode : the thread gathers the 8 corners of every level, blends them in
//            FP32 (Sec. 5.1, Eq. 11), appends the product-mode SH encodings
//            (Sec. 4.3), splits the values into 16-bit operand parts and
//            stores them into its lane of the activation columns (tcgen05.st).
//   layers : one elected thread issues tcgen05.mma kind::f16 with the
//            activations as the A operand in tensor memory and the weights as
//            the B operand in shared memory (M = 128, N = layer width, K in
//            steps of 16, FP32 accumulation) and commits to an mbarrier; every
//            thread reads its accumulator lane (tcgen05.ld), applies ReLU and
//            stores the next layer's operand parts.
//   decode : the last accumulator lane (4K FP32 raw outputs) in registers is
//            mapped (Table 1), sampled (Sec. 5.3) and evaluated (Eq. 4).
// Weights arrive once per CTA by a bulk asynchronous copy; the first tile is
// encoded meanwhile. Every wait on an mbarrier is bounded: on timeout the
// kernel records kStatusTimeout in the status word, drains what it has in
// flight (bounded), releases its tensor memory and returns.
//
// What bounds it on hash grids is the gathers: the L1 takes one request per
// lane and cycle, about 6 requests per level and query, and the L2 9.9 TB/s of
// random 32-byte sectors (0.64 to 0.83 of that reached). Activations in tensor
// memory leave shared memory to the weights alone, so the rest of the 256 KB
// stays L1 and four groups (16 warps, 128 registers) fit where activation
// tiles in shared memory left room for one to three. Measured against those
// (GB300, one call; in brackets with what followed: corner blocks, aligned
// pairs, elect_one): 64-wide product-mode network in the FP32-accuracy mode,
// 300,007 queries, 339 -> 140 us (107); paper-shaped hash grid, FP16,
// 2,073,600 queries, 869 -> 719 us (416); eight dense levels of four features,
// split BF16, 250,007 densities, 102 -> 72 us (57).
// Large batches read the dense levels through corner blocks (npm_tc.cuh), one
// or two 32-byte loads a level.
//
// FP32 models run here too, their values as three BF16 parts: 8 + 8 + 8 bits
// hold an FP32 value, and six products of parts leave out less than 2^-24 of
// it. Against the CUDA-core kernel (GB300): paper-shaped hash grid, 2^20
// queries, 717 -> 346 us, 3,001 log densities 31 -> 18 us; at 2^18 queries
// eight dense levels of four features 175 -> 76, 96-wide layers 303 -> 107,
// 128-wide 357 -> 124, sixteen lobes 258 -> 138, three features a level 173 ->
// 131, one level into 32-wide layers 47 -> 32 us. The error against
// FP64 stays where it was (density 3.6e-6 and 3.7e-6 relative, log density
// 2.7e-7 and 2.1e-7): the hardware exponentials decide it.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

#include <atomic>

#include "npm_kernels.h"
#include "npm_tc.cuh"

namespace npm {
namespace tc {

template <int OPS>
struct OpsTraits {
    // Parts of an activation and of a weight.
    static constexpr int parts = OPS == kThreeBf16 ? 3 : OPS == kOneBf16 || OPS == kOneFp16 ? 1 : 2;
    static constexpr int wparts = OPS == kThreeBf16 ? 3 : OPS == kOneBf16 ? 1 : 2;
    static constexpr bool fp32 = OPS == kTwoFp16 || OPS == kThreeBf16;  // FP32 grid table and sampler
    using GridT = typename std::conditional<fp32, float, __half>::type;
};

// Tile groups a CTA is compiled for: four at 128 registers; two for up to
// sixteen lobes, whose raw outputs alone take 64. FP32 on 2-feature grids also
// has an instance of three at 168 (launch_fwd_ops).
__host__ __device__ constexpr int fwd_groups(int kmax) { return kmax > 8 ? 2 : 4; }

// ----------------------------------------------------------- operands

// Three BF16 parts of a pair: each rounded to nearest from what the ones
// before leave, so that they add up to all 24 bits of the value. The first
// stays finite where a finite value would round to infinity.
//
// Infinite and NaN values: an infinite one has parts (largest, inf, NaN), so
// that every output of the row becomes NaN and, with the NaN kept by ReLU
// (relu_nan), the query's density NaN. FP32 arithmetic ends there too but for
// the cases in which ReLU takes infinity less infinity for zero. Where it takes
// a NaN weight's output, or those of a NaN input, for zero, so does this: the
// arrangement of the weights clears the rows of hidden layers that hold a NaN,
// and a row of inputs that holds one is cleared (clear_row).
__device__ __forceinline__ void three_bf16(float a, float b, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(p0) : "f"(b), "f"(a));
    a -= __uint_as_float(p0 << 16);
    b -= __uint_as_float(p0 & 0xffff0000u);
    p1 = pack_bf16(a, b);
    a -= __uint_as_float(p1 << 16);
    b -= __uint_as_float(p1 & 0xffff0000u);
    p2 = pack_bf16(a, b);
}
__device__ __forceinline__ float relu_nan(float a) {
    float d;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(d) : "f"(a));
    return d;
}
// NaN once a row of inputs has held one.
template <int OPS>
struct NanNote {
    float v;
    __device__ __forceinline__ void put(float a, float b) {
        if constexpr (OPS == kThreeBf16) asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(v) : "f"(a), "f"(b));
    }
};

// The operand parts of a pair of values (the first in the low half).
template <int OPS>
__device__ __forceinline__ void split_pair(float a, float b, uint32_t (&p)[OpsTraits<OPS>::parts]) {
    if constexpr (OPS == kOneFp16) {
        p[0] = pack_f16_sat(a, b);
    } else if constexpr (OPS == kOneBf16) {
        p[0] = pack_bf16(a, b);
    } else if constexpr (OPS == kTwoFp16) {
        p[0] = pack_f16_sat(a, b);
        p[1] = f16_residual(p[0], a, b);
    } else if constexpr (OPS == kThreeBf16) {
        three_bf16(a, b, p[0], p[1], p[2]);
    } else {
        p[0] = pack_bf16(a, b);
        p[1] = pack_bf16(a - __uint_as_float(p[0] << 16), b - __uint_as_float(p[0] & 0xffff0000u));
    }
}

// The same of max(a, 0), max(b, 0) (hidden layers). Split BF16 truncates the
// high part: the residual is then never negative and ReLU comes with both
// conversions.
template <int OPS>
__device__ __forceinline__ void relu_split_pair(float a, float b, uint32_t (&p)[OpsTraits<OPS>::parts]) {
    if constexpr (OPS == kOneFp16) {
        asm("cvt.rn.satfinite.relu.f16x2.f32 %0, %1, %2;" : "=r"(p[0]) : "f"(b), "f"(a));
    } else if constexpr (OPS == kOneBf16) {
        asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(p[0]) : "f"(b), "f"(a));
    } else if constexpr (OPS == kTwoFp16) {
        split_pair<OPS>(fmaxf(a, 0.0f), fmaxf(b, 0.0f), p);
    } else if constexpr (OPS == kThreeBf16) {
        split_pair<OPS>(relu_nan(a), relu_nan(b), p);
    } else {
        asm("cvt.rz.relu.bf16x2.f32 %0, %1, %2;" : "=r"(p[0]) : "f"(b), "f"(a));
        const float ra = a - __uint_as_float(p[0] << 16), rb = b - __uint_as_float(p[0] & 0xffff0000u);
        asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(p[1]) : "f"(rb), "f"(ra));
    }
}

// Where a thread's row of the activations goes: its lane of the tensor-memory
// columns, and (THIRD) its row of the third part's tile in shared memory, in
// planes (kPlane): four 64-wide groups' accumulators and two parts fill the 512
// columns.
template <bool THIRD>
struct ActRow {
    uint32_t tmem, part_cols;
    uint8_t* third;
};

// N operand pairs of this thread's row into the activation columns (two
// values each) col .. col + N of every part. All 32 lanes take part.
template <int OPS, bool THIRD, int N>
__device__ __forceinline__ void put_pairs(const ActRow<THIRD>& act, uint32_t col, const uint32_t (&v)[N][OpsTraits<OPS>::parts]) {
#pragma unroll
    for (int p = 0; p < OpsTraits<OPS>::parts; ++p) {
        if (THIRD && p == 2) {
            if constexpr (N == 8) {  // col is a multiple of 8
                uint8_t* at = act.third + (col >> 2) * kPlane;
                *reinterpret_cast<uint4*>(at) = make_uint4(v[0][p], v[1][p], v[2][p], v[3][p]);
                *reinterpret_cast<uint4*>(at + kPlane) = make_uint4(v[4][p], v[5][p], v[6][p], v[7][p]);
            } else {
#pragma unroll
                for (int i = 0; i < N; ++i)
                    *reinterpret_cast<uint32_t*>(act.third + ((col + i) >> 2) * kPlane + ((col + i) & 3u) * 4u) = v[i][p];
            }
            continue;
        }
        uint32_t r[N];
#pragma unroll
        for (int i = 0; i < N; ++i) r[i] = v[i][p];
        tmem_st(act.tmem + p * act.part_cols + col, r);
    }
}

// ------------------------------------------------------------- encode

// The grid table and, where a level has them, its corner blocks.
template <typename GT>
struct GridView {
    const GT* table;
    const uint4* blk;  // NULL: none
    uint32_t mask;     // levels with blocks
    __device__ __forceinline__ bool has(int l) const { return (mask >> l) & 1u; }
};

// Corner features of level l (2 features).
template <typename GT>
__device__ __forceinline__ void gather_level2(const TcCfg& tc, const GridView<GT>& grid, int l, const Cell& cl,
                                              Level2<GT>& v) {
    const DevCfg& cfg = tc.base;
    if (grid.has(l)) {
        const uint32_t D = (uint32_t)cfg.level_res[l];
        v.load_blocks(grid.blk, tc.blk_off[l] + corner_idx1(cfg, l, cl, 0), D * D);
    } else {
        v.load_table(cfg, grid.table, l, cl);
    }
}

// Features 4h .. 4h + 3 of a level of F = 4 or 8 features (blocks: F = 4).
template <typename GT>
__device__ __forceinline__ float4 blend_level4(const TcCfg& tc, const GridView<GT>& grid, int l, const Cell& cl, int F,
                                               int h) {
    const DevCfg& cfg = tc.base;
    decltype(load_raw4(grid.table, 0u, F, 0)) raw[8];
    if (grid.has(l)) {
        const uint32_t D = (uint32_t)cfg.level_res[l];
        gather_blocks4(grid.blk, tc.blk_off[l] + corner_idx1(cfg, l, cl, 0), D, D * D, grid.table, raw);
    } else {
        const GT* g = grid.table + (size_t)cfg.level_off[l] * F;
        uint32_t idx[8];
        corner_idx8(cfg, l, cl, idx);
#pragma unroll
        for (int c = 0; c < 8; ++c) raw[c] = load_raw4(g, idx[c], F, h);
    }
    float w[8];
    corner_w8(cl, w);
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float4 v = widen4(raw[c]);
        a.x = fmaf(w[c], v.x, a.x);
        a.y = fmaf(w[c], v.y, a.y);
        a.z = fmaf(w[c], v.z, a.z);
        a.w = fmaf(w[c], v.w, a.w);
    }
    return a;
}

// Values of a row one after another, stored in pairs.
template <int OPS, bool THIRD>
struct RowPacker {
    ActRow<THIRD> act;
    NanNote<OPS>& nan;
    int k;
    float prev;
    __device__ __forceinline__ void put(float v) {
        if (k & 1) {
            uint32_t p[1][OpsTraits<OPS>::parts];
            nan.put(prev, v);
            split_pair<OPS>(prev, v, p[0]);
            __syncwarp();
            put_pairs<OPS, THIRD, 1>(act, (uint32_t)(k >> 1), p);
        }
        prev = v;
        ++k;
    }
};

// Product-mode inputs of query j (Sec. 4.3): SH of the outgoing direction and
// of the normal, roughness.
__device__ __forceinline__ void product_inputs(const QuerySeg& S, uint32_t j, bool valid, float (&e)[22]) {
    float ax[7] = {0.0f, 0.0f, 1.0f, 0.0f, 0.0f, 1.0f, 0.0f};
    if (valid)
#pragma unroll
        for (int i = 0; i < 7; ++i) ax[i] = S.aux[i * S.ld + j];
    __syncwarp();
    sh_band4(ax[0], ax[1], ax[2], e);
    sh_band2(ax[3], ax[4], ax[5], e + 16);
    e[20] = ax[6];
    e[21] = 0.0f;
}

// The network input of query j at (x, y, z) in the unit box: this thread's row of the activation
// columns, padded with zeros to the layer's kp values. FEAT: features per
// level (2 or 4), or 0 for any.
template <int FEAT, int OPS, int NF, bool THIRD>
__device__ __forceinline__ void encode_row(const TcCfg& tc, const GridView<typename OpsTraits<OPS>::GridT>& grid,
                                           float x, float y, float z, const QuerySeg& S, uint32_t j, bool valid,
                                           const ActRow<THIRD>& act, NanNote<OPS>& nan) {
    const DevCfg& cfg = tc.base;
    constexpr int P = OpsTraits<OPS>::parts;
    __syncwarp();
    const int L = cfg.n_levels, F = FEAT ? FEAT : cfg.feat;
    if constexpr (FEAT == 2) {
        // NF levels' gathers in flight before the first is blended.
        int l = 0;
        for (; l + NF <= L; l += NF) {
            Cell cl[NF];
            Level2<typename OpsTraits<OPS>::GridT> v[NF];
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                cl[i] = make_cell_in(x, y, z, cfg.level_res[l + i]);
                gather_level2(tc, grid, l + i, cl[i], v[i]);
            }
            uint32_t p[NF][P];
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const float2 a = v[i].blend(cl[i]);
                nan.put(a.x, a.y);
                split_pair<OPS>(a.x, a.y, p[i]);
            }
            put_pairs<OPS, THIRD, NF>(act, (uint32_t)l, p);
        }
        for (; l < L; ++l) {
            const Cell cl = make_cell_in(x, y, z, cfg.level_res[l]);
            Level2<typename OpsTraits<OPS>::GridT> v;
            gather_level2(tc, grid, l, cl, v);
            const float2 a = v.blend(cl);
            uint32_t p[1][P];
            nan.put(a.x, a.y);
            split_pair<OPS>(a.x, a.y, p[0]);
            put_pairs<OPS, THIRD, 1>(act, (uint32_t)l, p);
        }
    } else if (FEAT == 4 || F == 4 || F == 8) {
#pragma unroll(FEAT == 4 ? 2 : 1)
        for (int l = 0; l < L; ++l) {
            const Cell cl = make_cell_in(x, y, z, cfg.level_res[l]);
            for (int h = 0; h < (F >> 2); ++h) {
                const float4 a = blend_level4(tc, grid, l, cl, F, h);
                uint32_t p[2][P];
                nan.put(a.x, a.y);
                nan.put(a.z, a.w);
                split_pair<OPS>(a.x, a.y, p[0]);
                split_pair<OPS>(a.z, a.w, p[1]);
                put_pairs<OPS, THIRD, 2>(act, (uint32_t)((l * F + 4 * h) >> 1), p);
            }
        }
    } else {
        RowPacker<OPS, THIRD> row{act, nan, 0, 0.0f};
        for (int l = 0; l < L; ++l) {
            const Cell cl = make_cell_in(x, y, z, cfg.level_res[l]);
            if (F == 2) {
                Level2<typename OpsTraits<OPS>::GridT> v;
                gather_level2(tc, grid, l, cl, v);
                const float2 a = v.blend(cl);
                row.put(a.x);
                row.put(a.y);
            } else {  // one, or another number that no vector load fits
                const auto* g = grid.table + (size_t)cfg.level_off[l] * F;
                uint32_t idx[8];
                float w[8];
                corners8(cfg, l, cl, idx, w);
                for (int f = 0; f < F; ++f) {
                    float s = 0.0f;
#pragma unroll
                    for (int c = 0; c < 8; ++c) s = fmaf(w[c], load_feat(g + (size_t)idx[c] * F, f), s);
                    row.put(s);
                }
            }
        }
        if (cfg.mode != NPM_PRODUCT && (row.k & 1)) row.put(0.0f);
        if (cfg.mode == NPM_PRODUCT) {
            float e[22];
            product_inputs(S, j, valid, e);
#pragma unroll
            for (int i = 0; i < 21; ++i) row.put(e[i]);
            if (row.k & 1) row.put(0.0f);
        }
    }
    uint32_t col = (uint32_t)(cfg.grid_feats + 1) >> 1;
    if (cfg.mode == NPM_PRODUCT) {
        if (FEAT != 0 || F == 4 || F == 8) {
            // An even number of grid features: 21 values and one zero.
            float e[22];
            product_inputs(S, j, valid, e);
#pragma unroll
            for (int i = 0; i < 22; i += 2) {
                uint32_t p[1][P];
                nan.put(e[i], e[i + 1]);
                split_pair<OPS>(e[i], e[i + 1], p[0]);
                put_pairs<OPS, THIRD, 1>(act, col + (uint32_t)(i >> 1), p);
            }
        }
        col = (uint32_t)(cfg.grid_feats + 22) >> 1;
    }
    const uint32_t end = (uint32_t)tc.layer[0].Kp >> 1;
    for (; col < end; ++col) {
        const uint32_t p[1][P] = {};
        put_pairs<OPS, THIRD, 1>(act, col, p);
    }
}

// This thread's row of the first layer's input set to zero where `clear`. All
// 32 lanes take part; rare.
template <int OPS, bool THIRD>
__device__ __noinline__ void clear_row(const TcCfg& tc, const ActRow<THIRD> act, bool clear) {
    const uint32_t keep = clear ? 0u : ~0u;
    tmem_wait_st();
    for (uint32_t col = 0; col < (uint32_t)tc.layer[0].Kp >> 1; col += 2) {
#pragma unroll
        for (int p = 0; p < OpsTraits<OPS>::parts; ++p) {
            if (THIRD && p == 2) {
                uint2* at = reinterpret_cast<uint2*>(act.third + (col >> 2) * kPlane + (col & 3u) * 4u);
                *at = make_uint2(at->x & keep, at->y & keep);
                continue;
            }
            uint32_t r[2];
            tmem_ld2(act.tmem + p * act.part_cols + col, r);
            tmem_wait2(r);
            r[0] &= keep;
            r[1] &= keep;
            tmem_st(act.tmem + p * act.part_cols + col, r);
        }
    }
}

// --------------------------------------------------------------- decode

// Two lobes decoded (Table 1) for the density in packed FP32, two lobes an
// instruction, in the arithmetic of decode_lobe_fast, vmf_scaled_norm_fast and
// vmf_eval_fast: hardware exponential, logarithm, reciprocal, sine and cosine
// on arguments in their accurate ranges. theta = pi s(t'), phi = pi + ph with
// ph = pi (2 s(p') - 1); the mean is (-nx, -ny, -nz).
struct LobePair2 {
    float2 kap, th, ph, nx, ny, nz;

    template <typename Raw>
    __device__ __forceinline__ void decode(int kappa_act, const Raw& raw, int i) {
        const float2 rk = make_float2(raw(4 * i + 1), raw(4 * i + 5)), rt = make_float2(raw(4 * i + 2), raw(4 * i + 6)),
                     rp = make_float2(raw(4 * i + 3), raw(4 * i + 7));
        if (kappa_act == NPM_EXP) {
            const float2 e = __fmul2_rn(rk, f2(kL2E));
            kap = make_float2(hw_ex2_tiny(e.x), hw_ex2_tiny(e.y));
        } else {
            // max(t, 0) + ln(1 + e^{-|t|})
            const float2 e = __fmul2_rn(make_float2(fabsf(rk.x), fabsf(rk.y)), f2(-kL2E));
            const float2 q = __fadd2_rn(make_float2(hw_ex2(e.x), hw_ex2(e.y)), f2(1.0f));
            kap = __ffma2_rn(make_float2(hw_lg2(q.x), hw_lg2(q.y)), f2(kLn2),
                             make_float2(fmaxf(rk.x, 0.0f), fmaxf(rk.y, 0.0f)));
        }
        const float2 st = logistic2(rt), sp = logistic2(rp);
        th = __fmul2_rn(st, f2(kPi));
        ph = __fmul2_rn(__ffma2_rn(sp, f2(2.0f), f2(-1.0f)), f2(kPi));
        const float2 a = __fadd2_rn(th, f2(-0.5f * kPi));  // sin(th) = cos(a), cos(th) = -sin(a)
        float sa0, ca0, sa1, ca1, sb0, cb0, sb1, cb1;
        __sincosf(a.x, &sa0, &ca0);
        __sincosf(a.y, &sa1, &ca1);
        __sincosf(ph.x, &sb0, &cb0);
        __sincosf(ph.y, &sb1, &cb1);
        const float2 sth = make_float2(ca0, ca1);
        nx = __fmul2_rn(sth, make_float2(cb0, cb1));
        ny = __fmul2_rn(sth, make_float2(sb0, sb1));
        nz = make_float2(sa0, sa1);
    }
    __device__ __forceinline__ static float2 logistic2(float2 t) {
        const float2 e = __fmul2_rn(t, f2(-kL2E));
        const float2 q = __fadd2_rn(make_float2(hw_ex2(e.x), hw_ex2(e.y)), f2(1.0f));
        return make_float2(hw_rcp(q.x), hw_rcp(q.y));
    }
    // kappa (mu . w - 1) log2(e)
    __device__ __forceinline__ float2 exponent(const float (&w)[3]) const {
        const float2 d = __ffma2_rn(nz, f2(w[2]), __ffma2_rn(ny, f2(w[1]), __fmul2_rn(nx, f2(w[0]))));  // -mu . w
        return __fmul2_rn(__fmul2_rn(kap, __fadd2_rn(d, f2(1.0f))), f2(-kL2E));
    }
    // c(kappa) = kappa / (2 pi (1 - e^{-2 kappa}))
    __device__ __forceinline__ float2 norm() const {
        const float2 k = kap;
        float2 s = __ffma2_rn(k, f2(4.0f / 15.0f), f2(-2.0f / 3.0f));
        s = __ffma2_rn(k, s, f2(4.0f / 3.0f));
        s = __ffma2_rn(k, s, f2(-2.0f));
        s = __fmul2_rn(k, __ffma2_rn(k, s, f2(2.0f)));
        const float2 x = __fmul2_rn(k, f2(-2.0f * kL2E));
        const float2 e = __ffma2_rn(make_float2(hw_ex2(x.x), hw_ex2(x.y)), f2(-1.0f), f2(1.0f));
        const float2 em = __fmul2_rn(make_float2(k.x < 0.05f ? s.x : e.x, k.y < 0.05f ? s.y : e.y), f2(2.0f * kPi));
        const float2 c = __fmul2_rn(k, make_float2(hw_rcp(em.x), hw_rcp(em.y)));
        const float2 c0 = __ffma2_rn(k, f2(kInv4Pi), f2(kInv4Pi));  // kappa -> 0
        return make_float2(k.x < 1e-6f ? c0.x : c.x, k.y < 1e-6f ? c0.y : c.y);
    }
};

// Table 1, sampling (Sec. 5.3) and density (Eq. 4) of one query from its raw
// outputs. Only the chosen lobe is decoded for the sample; the density then
// decodes pair by pair, so that no array of decoded lobes stays live (nine
// lobe decodes instead of eight, half the registers). Pairs past the last
// lobe read the zeros of the padded last layer.
// u: uniforms when sampling, direction when evaluating.
template <int KMAX, bool FP32>
__device__ __forceinline__ void decode_row(const DevCfg& cfg, const uint32_t (&rawu)[KMAX / 4][16], const QuerySeg& S,
                                           uint32_t j, bool valid, const float (&u)[4], bool sample, bool log_pdf) {
    const int K = cfg.K;
    auto raw = [&](int i) { return __uint_as_float(rawu[i >> 4][i & 15]); };
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
        if (i < K) mx = fmaxf(mx, raw(4 * i));
    float lam[KMAX], ssum = 0.0f;
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
        if (i < K) {
            lam[i] = __expf(raw(4 * i) - mx);
            ssum += lam[i];
        }
    const float inv = __fdividef(1.0f, ssum);  // ssum in [1, K]
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
        if (i < K) lam[i] *= inv;
    float w[3] = {u[0], u[1], u[2]};
    if (sample) {
        // Smallest lobe i with u0 < lambda_0 + ... + lambda_i (last if none).
        float cum = 0.0f, rk = raw(1), rt = raw(2), rp = raw(3);
        bool found = false;
#pragma unroll
        for (int i = 0; i < KMAX; ++i)
            if (i < K) {
                cum += lam[i];
                if (!found) {
                    rk = raw(4 * i + 1);
                    rt = raw(4 * i + 2);
                    rp = raw(4 * i + 3);
                }
                found = found || u[0] < cum;
            }
        if (S.ufrac > 0.0f && u[3] < S.ufrac) {
            uniform_sphere(u[1], u[2], w);
        } else {
            Lobe sl;
            decode_lobe_fast(cfg.kappa_act, rk, rt, rp, sl, nullptr, nullptr);
            if (FP32) vmf_sample(sl, u[1], u[2], w);
            else vmf_sample_rp(sl, u[1], u[2], w);
        }
    }
    float pv = 0.0f;
    if (!sample && log_pdf) {
        // log V (Eq. 4 in log-sum-exp form), the weights' logs taken from the
        // logits so that they stay finite where lambda_i underflows.
        const float lnorm = mx + __logf(ssum);
        float m = -INFINITY;
#pragma unroll
        for (int i = 0; i < KMAX; i += 2)
            if (i < K) {
                LobePair2 p;
                p.decode(cfg.kappa_act, raw, i);
                const float2 e = p.exponent(w), c = p.norm();
                lam[i] = (raw(4 * i) - lnorm) + kLn2 * (hw_lg2(c.x) + e.x);
                m = fmaxf(m, lam[i]);
                lam[i + 1] = -INFINITY;
                if (i + 1 < K) lam[i + 1] = (raw(4 * i + 4) - lnorm) + kLn2 * (hw_lg2(c.y) + e.y);
                m = fmaxf(m, lam[i + 1]);
            }
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < KMAX; ++i)
            if (i < K) s += __expf(lam[i] - m);
        pv = m + __logf(s);
    } else {
#pragma unroll
        for (int i = 0; i < KMAX; i += 2)
            if (i < K) {
                LobePair2 p;
                p.decode(cfg.kappa_act, raw, i);
                const bool two = i + 1 < K;
                const float2 l = make_float2(lam[i], two ? lam[i + 1] : 0.0f);
                if (S.mix && valid) {
                    float* mo = S.mix + (int64_t)(4 * i) * S.ld + j;
                    mo[0] = l.x;
                    mo[S.ld] = p.kap.x;
                    mo[2 * S.ld] = p.th.x;
                    mo[3 * S.ld] = p.ph.x + kPi;
                    if (two) {
                        mo += 4 * S.ld;
                        mo[0] = l.y;
                        mo[S.ld] = p.kap.y;
                        mo[2 * S.ld] = p.th.y;
                        mo[3 * S.ld] = p.ph.y + kPi;
                    }
                }
                const float2 e = p.exponent(w);
                const float2 v = __fmul2_rn(l, __fmul2_rn(p.norm(), make_float2(hw_ex2_tiny(e.x), hw_ex2_tiny(e.y))));
                pv += v.x;
                if (two) pv += v.y;
            }
        if (sample && S.ufrac > 0.0f) pv = S.ufrac * kInv4Pi + (1.0f - S.ufrac) * pv;
    }
    if (valid) {
        if (sample) {
            S.dir[j] = w[0];
            S.dir[S.ld + j] = w[1];
            S.dir[2 * S.ld + j] = w[2];
        }
        S.pdf[j] = pv;
    }
}

// Warp-per-query form of the decode, sample and density (Table 1, Sec. 5.3,
// Eq. 4): lane l of a warp owns lobe l mod KMAX of one query, so a warp
// serves 32 / KMAX queries per pass and KMAX passes cover its 32 rows. The
// raw outputs of the tile are staged in shared memory (row stride 4 KMAX + 4
// floats keeps both the row writes and the lobe reads free of bank
// conflicts). Softmax and density are reductions over the query's lanes;
// the lobe choice takes the running sum of the weights in lobe order (a
// serial scan, the same rounding as the thread-per-row form) and a ballot;
// every lane samples its own lobe and the chosen lane's direction is
// broadcast. Slower than decode_row (one thread per query), so a tuning override
// selects it: split BF16, paper-shaped grid, 1.60 against 1.96 G queries/s.
template <int KMAX>
__device__ __forceinline__ void tc_decode_warp(const TcCfg& tc, const float* __restrict__ sRaw, int warp, int lane,
                                               int64_t j0, int64_t n, int64_t ld, const float* __restrict__ uin,
                                               float ufrac, bool sample, float* __restrict__ dir_out,
                                               float* __restrict__ pdf_out, float* __restrict__ mix_out,
                                               bool log_pdf) {
    constexpr int RS = 4 * KMAX + 4;
    constexpr int QP = 32 / KMAX;  // queries per pass
    constexpr unsigned kAll = 0xffffffffu;
    const DevCfg& cfg = tc.base;
    const int K = cfg.K;
    const int i = lane & (KMAX - 1);
    const int qsub = lane / KMAX;
    const unsigned seg = KMAX == 32 ? kAll : (((1u << KMAX) - 1u) << (qsub * KMAX));
    const bool act = i < K;
#pragma unroll 1
    for (int p = 0; p < KMAX; ++p) {
        const int r = warp * 32 + p * QP + qsub;
        const int64_t j = j0 + r;
        const bool valid = j < n;
        const float4 rv = *reinterpret_cast<const float4*>(sRaw + r * RS + 4 * i);
        float mx = act ? rv.x : -INFINITY;
#pragma unroll
        for (int o = 1; o < KMAX; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(kAll, mx, o));
        const float e = act ? __expf(rv.x - mx) : 0.0f;
        float ssum = e;
#pragma unroll
        for (int o = 1; o < KMAX; o <<= 1) ssum += __shfl_xor_sync(kAll, ssum, o);
        Lobe L;
        L.lam = e * __fdividef(1.0f, ssum);
        float th, ph;
        decode_lobe_fast(cfg.kappa_act, rv.y, rv.z, rv.w, L, &th, &ph);
        const float cn = vmf_scaled_norm_fast(L.kap);
        if (mix_out && valid && act) {
            mix_out[(4 * i + 0) * ld + j] = L.lam;
            mix_out[(4 * i + 1) * ld + j] = L.kap;
            mix_out[(4 * i + 2) * ld + j] = th;
            mix_out[(4 * i + 3) * ld + j] = ph;
        }
        float w[3] = {0.0f, 0.0f, 1.0f};
        bool uni = false;
        if (sample) {
            float u0 = 0.0f, u1 = 0.0f, u2 = 0.0f;
            if (valid) {
                u0 = uin[j];
                u1 = uin[ld + j];
                u2 = uin[2 * ld + j];
                uni = ufrac > 0.0f && uin[3 * ld + j] < ufrac;
            }
            // Running sum of the weights in lobe order.
            float cum = i == 0 ? L.lam : 0.0f;
#pragma unroll
            for (int k = 1; k < KMAX; ++k) {
                const float prev = __shfl_up_sync(kAll, cum, 1);
                if (i == k) cum = prev + L.lam;
            }
            const unsigned hit = __ballot_sync(kAll, act && u0 < cum) & seg;
            const int sel = hit ? __ffs(hit) - 1 - qsub * KMAX : K - 1;
            float d[3];
            if (uni) uniform_sphere(u1, u2, d);
            else vmf_sample_rp(L, u1, u2, d);
#pragma unroll
            for (int a = 0; a < 3; ++a) w[a] = __shfl_sync(kAll, d[a], qsub * KMAX + sel);
        } else if (valid) {
            w[0] = uin[j];
            w[1] = uin[ld + j];
            w[2] = uin[2 * ld + j];
        }
        float pv;
        if (!sample && log_pdf) {
            const float dd = L.mu[0] * w[0] + L.mu[1] * w[1] + L.mu[2] * w[2];
            const float a = act ? (rv.x - mx) - __logf(ssum) + __logf(cn) + L.kap * (dd - 1.0f) : -INFINITY;
            float m = a;
#pragma unroll
            for (int o = 1; o < KMAX; o <<= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
            float sx = act ? __expf(a - m) : 0.0f;
#pragma unroll
            for (int o = 1; o < KMAX; o <<= 1) sx += __shfl_xor_sync(kAll, sx, o);
            pv = m + __logf(sx);
        } else {
            pv = act ? L.lam * vmf_eval_fast(L, cn, w[0], w[1], w[2]) : 0.0f;
#pragma unroll
            for (int o = 1; o < KMAX; o <<= 1) pv += __shfl_xor_sync(kAll, pv, o);
            if (sample && ufrac > 0.0f) pv = ufrac * kInv4Pi + (1.0f - ufrac) * pv;
        }
        if (valid && i == 0) {
            if (sample) {
                dir_out[j] = w[0];
                dir_out[ld + j] = w[1];
                dir_out[2 * ld + j] = w[2];
            }
            pdf_out[j] = pv;
        }
    }
}

// --------------------------------------------------------------- kernel

// Bytes of a group's third activation part in shared memory.
template <bool THIRD>
__host__ __device__ inline uint32_t fwd_third_bytes(const TcCfg& tc) {
    return THIRD ? tc.a_cols / 4u * kPlane : 0u;
}

// The MMAs of one layer: every K step of each product of parts, the smallest
// products first, so that the large ones meet the accumulator's rounding only
// Kp / 16 times. Issued by one thread.
template <int OPS, bool THIRD>
__device__ __forceinline__ void issue_layer(const TcCfg& tc, const TcLayer& ly, uint32_t acc, uint32_t act,
                                            uint32_t third, uint32_t sW_addr) {
    const uint64_t b0 = umma_desc(sW_addr + ly.w_off, 128u, (uint32_t)(ly.Kp >> 3) * 128u);
    with_steps(ly.Kp >> 4, [&](auto steps) {
        constexpr int NK = decltype(steps)::count;
        const int nk = NK ? NK : ly.Kp >> 4;
        bool first = true;
        auto product = [&](int ap, int wp) {
            const uint64_t b = b0 + (uint64_t)wp * (tc.w_bytes >> 4);
            const uint32_t a = act + (uint32_t)ap * tc.a_cols;
            mma_tmem_a(acc, a, b, ly.idesc, first ? 0u : 1u);
            first = false;
#pragma unroll(NK ? NK : 1)
            for (int s = 1; s < nk; ++s) mma_tmem_a(acc, a + 8u * (uint32_t)s, b + (uint64_t)(16 * s), ly.idesc, 1u);
        };
        if constexpr (OPS == kThreeBf16) {
            // (1, 2), (2, 1) and (2, 2) lie 2^-26 and more below the product.
            product(0, 2);
            if constexpr (THIRD) {
                const uint64_t a2 = umma_desc(third, kPlane, 128u);
#pragma unroll(NK ? NK : 1)
                for (int s = 0; s < nk; ++s)
                    mma_bf16(acc, a2 + (uint64_t)(2 * (kPlane >> 4) * s), b0 + (uint64_t)(16 * s), ly.idesc, 1u);
            } else {
                product(2, 0);
            }
            product(1, 1);
        }
        if constexpr (OpsTraits<OPS>::parts >= 2) product(1, 0);
        if constexpr (OpsTraits<OPS>::wparts >= 2) product(0, 1);
        product(0, 0);
    });
}

// WARPDEC: the warp-per-query decode (tc_decode_warp) from raw outputs staged
// in shared memory. THIRD: the third activation part lies in shared memory.
template <int KMAX, int FEAT, int OPS, bool WARPDEC = false, int GMAX = fwd_groups(KMAX),
          bool THIRD = (OPS == kThreeBf16)>
__global__ void __launch_bounds__(kThreads * GMAX, 1)
    k_forward_tc(const __grid_constant__ TcCfg tc, const typename OpsTraits<OPS>::GridT* __restrict__ table,
                 const uint4* blk, const uint8_t* __restrict__ wblob, const __grid_constant__ QueryBatch qb,
                 int* __restrict__ status, long long wait_limit) {
    extern __shared__ __align__(1024) uint8_t smem[];
    // Levels of 2-feature grids gathered before the first is blended: what the
    // registers hold without spilling (GB300, 2^20 queries of the paper-shaped
    // grid: FP16 with 2, 3, 4: 241, 229, 241 us; split BF16 254, 247, 256;
    // FP32 accuracy with 1, 2: 312, 324; FP32 in three groups with 1, 2, 3:
    // 369, 345, 348).
    constexpr int NF = GMAX == 3 ? 2 : OpsTraits<OPS>::fp32 ? 1 : 3;
    const int G = (int)(blockDim.x >> 7);
    const int g = (int)warp_uniform(threadIdx.x >> 7);  // tile group
    const int t = (int)(threadIdx.x & 127);             // row of the group's tile
    const int warp = (int)warp_uniform((threadIdx.x >> 5) & 3u);                 // warp of the group (its tensor-memory lane quarter)
    const uint32_t wbytes = (uint32_t)OpsTraits<OPS>::wparts * tc.w_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + wbytes);  // [0] weights, [1 + g] MMAs
    uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 1 + G);
    const uint32_t bar_w = smem_u32(&bars[0]), bar_mma = smem_u32(&bars[1 + g]);
    uint32_t cta_cols = 32;
    while (cta_cols < (uint32_t)G * tc.g_cols) cta_cols <<= 1;

    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(cta_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        for (int i = 0; i <= G; ++i) mbar_init(smem_u32(&bars[i]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_w), "r"(wbytes) : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                smem_u32(smem)),
            "l"(wblob), "r"(wbytes), "r"(bar_w)
            : "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // This group's columns: the accumulator, then the activations' parts; the
    // third part's tile.
    const uint32_t acc = warp_uniform(*tslot) + (uint32_t)g * tc.g_cols, act = acc + tc.d_cols;
    uint8_t* third = smem + fwd_stage_off(wbytes, G) + (uint32_t)g * fwd_third_bytes<THIRD>(tc);
    const uint32_t lanes = (uint32_t)(warp * 32) << 16;
    const ActRow<THIRD> row{act + lanes, tc.a_cols, third + t * 16};
    const uint32_t sW_addr = smem_u32(smem);
    const int L = tc.base.n_layers;
    const bool sample = qb.sample != 0;
    // Launched as a programmatic dependent (of the corner blocks' check), the
    // steps above overlap that kernel, which writes the blocks alone.
    grid_dep_wait();
    const GridView<typename OpsTraits<OPS>::GridT> grid{table, blk, blk ? tc.blk_mask : 0u};

    // Tiles and queries of a segment in 32 bits: batches hold at most 2^31
    // queries.
    uint32_t ntiles = (uint32_t)qb.total_tiles, n0 = (uint32_t)qb.seg[0].n;
    if (qb.n_dev) {
        n0 = (uint32_t)*qb.n_dev;
        ntiles = (n0 + (kTile - 1)) / kTile;
    }
    bool ok = true, issued = false;
    uint32_t phase = 0;
    // Tiles are dealt to the CTAs first and to a CTA's groups second, so a
    // batch of fewer tiles than groups spreads over as many SMs as it can.
    const uint32_t stride = gridDim.x * (uint32_t)G;
    for (uint32_t tile = blockIdx.x + (uint32_t)g * gridDim.x; tile < ntiles; tile += stride) {
        int sg = 0;
        while (sg + 1 < qb.nseg && tile >= (uint32_t)qb.seg[sg + 1].tile0) ++sg;
        const QuerySeg& S = qb.seg[sg];
        const uint32_t n = (sg == 0 && qb.n_dev) ? n0 : (uint32_t)S.n;
        const uint32_t base = (tile - (uint32_t)S.tile0) * kTile, j = base + t;
        const bool valid = j < n;
        float x = 0.0f, y = 0.0f, z = 0.0f;
        if (valid) {
            x = clamp01(S.pos[j]);
            y = clamp01(S.pos[S.ld + j]);
            z = clamp01(S.pos[2 * S.ld + j]);
        }
        if (warp == 3) {
            // The group's next tile's positions into L2 (three 512-byte rows).
            const int lane = t & 31, r = lane >> 2;
            const uint32_t nt = tile + stride;
            if (r < 3 && nt < ntiles) {
                int s2 = sg;
                while (s2 + 1 < qb.nseg && nt >= (uint32_t)qb.seg[s2 + 1].tile0) ++s2;
                const QuerySeg& S2 = qb.seg[s2];
                const uint32_t b2 = (nt - (uint32_t)S2.tile0) * kTile + 32 * (lane & 3);
                const uint32_t n2 = (s2 == 0 && qb.n_dev) ? n0 : (uint32_t)S2.n;
                if (b2 < n2) asm volatile("prefetch.global.L2 [%0];" ::"l"(S2.pos + r * S2.ld + b2));
            }
        }
        NanNote<OPS> nan{0.0f};
        encode_row<FEAT, OPS, NF, THIRD>(tc, grid, x, y, z, S, j, valid, row, nan);
        if constexpr (OPS == kThreeBf16)
            if (L > 1 && __any_sync(0xffffffffu, isnan(nan.v))) clear_row<OPS, THIRD>(tc, row, isnan(nan.v));
        // The uniforms (or the direction), loaded now so that their latency
        // passes during the layers.
        float u[4] = {0.0f, 0.0f, sample ? 0.0f : 1.0f, 0.0f};
        if (valid) {
            u[0] = S.uin[j];
            u[1] = S.uin[S.ld + j];
            u[2] = S.uin[2 * S.ld + j];
            if (S.ufrac > 0.0f) u[3] = S.uin[3 * S.ld + j];
        }
        __syncwarp();
        tmem_wait_st();
        if constexpr (THIRD) fence_async_smem();
        tc_fence_before();
        if (tc_group_sync_or(g, !ok)) {
            ok = false;
            break;
        }
        uint32_t raw[KMAX / 4][16];
        for (int l = 0; l < L; ++l) {
            const TcLayer& ly = tc.layer[l];
            if (warp == 0) {
                // The weights have arrived (once per CTA).
                if (!issued) ok = __all_sync(0xffffffffu, mbar_wait_limit(bar_w, 0, wait_limit));
                if (ok) {
                    tc_fence_after();
                    if (elect_one()) {
                        issue_layer<OPS, THIRD>(tc, ly, acc, act, smem_u32(third), sW_addr);
                        mma_commit(bar_mma);
                    }
                    __syncwarp();
                    issued = true;
                }
            }
            // Every warp waits on the MMAs' barrier; a wait that gives up is
            // made known to the group at its next barrier.
            ok = __all_sync(0xffffffffu, ok && mbar_wait_limit(bar_mma, phase, wait_limit));
            phase ^= 1u;
            tc_fence_after();
            if (l < L - 1) {
                if (ok) {
#pragma unroll 2
                    for (int c0 = 0; c0 < ly.Np; c0 += 16) {
                        uint32_t r[16];
                        tmem_ld16(acc + lanes + (uint32_t)c0, r);
                        tmem_wait16(r);
                        uint32_t p[8][OpsTraits<OPS>::parts];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            relu_split_pair<OPS>(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]), p[i]);
                        put_pairs<OPS, THIRD, 8>(row, (uint32_t)(c0 >> 1), p);
                    }
                    tmem_wait_st();
                }
                if constexpr (THIRD) fence_async_smem();
                tc_fence_before();
                if (tc_group_sync_or(g, !ok)) {
                    ok = false;
                    break;
                }
            } else if (ok) {
#pragma unroll
                for (int c = 0; c < KMAX / 4; ++c)
                    if (c * 16 < ly.Np) tmem_ld16(acc + lanes + (uint32_t)(c * 16), raw[c]);
#pragma unroll
                for (int c = 0; c < KMAX / 4; ++c)
                    if (c * 16 < ly.Np) tmem_wait16(raw[c]);
                tc_fence_before();
            }
        }
        if constexpr (WARPDEC) {
            // Stage the raw outputs, then decode a query per 32 / KMAX lanes.
            constexpr int RS = 4 * KMAX + 4;
            float* sRaw = reinterpret_cast<float*>(smem + fwd_stage_off(wbytes, G)) + g * kTile * RS;
            if (tc_group_sync_or(g, !ok)) {
                ok = false;
                break;
            }
#pragma unroll
            for (int c = 0; c < KMAX / 4; ++c)
                if (c * 16 < tc.layer[L - 1].Np)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        *reinterpret_cast<uint4*>(sRaw + t * RS + 16 * c + 4 * i) =
                            make_uint4(raw[c][4 * i], raw[c][4 * i + 1], raw[c][4 * i + 2], raw[c][4 * i + 3]);
            tc_group_sync(g);
            tc_decode_warp<KMAX>(tc, sRaw, warp, t & 31, base, n, S.ld, S.uin, S.ufrac, sample, S.dir, S.pdf, S.mix,
                                 qb.log_pdf != 0);
        } else {
            if (ok)
                decode_row<KMAX, OpsTraits<OPS>::fp32>(tc.base, raw, S, j, valid, u, sample, qb.log_pdf != 0);
        }
    }
    if (!ok && (t & 31) == 0) atomicOr(status, kStatusTimeout);
    // Before the tensor and shared memory are released: whatever a wait gave
    // up on and may still be in flight (the weights' bulk copy; this group's
    // last MMAs, of the phase before `phase`), again with a bound.
    if (threadIdx.x == 32) (void)mbar_wait_bounded(bar_w, 0);
    if (t == 0 && !ok && issued) (void)mbar_wait_bounded(bar_mma, phase ^ 1u);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tslot), "r"(cta_cols) : "memory");
    }
}

// ------------------------------------------------------------- launcher

// Columns of a tile group, and the groups of a CTA: as many as the instance is
// compiled for and the 512 tensor-memory columns and the shared memory hold.
template <int OPS, bool THIRD>
uint32_t fwd_group_cols(const TcCfg& c) {
    return c.d_cols + (uint32_t)(OpsTraits<OPS>::parts - (THIRD ? 1 : 0)) * c.a_cols;
}
template <int OPS, bool THIRD>
int fwd_group_count(const TcCfg& c, int most) {
    const uint32_t wbytes = (uint32_t)OpsTraits<OPS>::wparts * c.w_bytes;
    int G = most;
    while (G > 1 && ((uint32_t)G * fwd_group_cols<OPS, THIRD>(c) > 512u ||
                     fwd_stage_off(wbytes, G) + (uint32_t)G * fwd_third_bytes<THIRD>(c) > 226u * 1024u))
        --G;
    return G;
}

template <int KMAX, int FEAT, int OPS, bool WARPDEC = false, int GMAX = fwd_groups(KMAX),
          bool THIRD = (OPS == kThreeBf16)>
cudaError_t launch_fwd(const TcCfg& cfg, const void* grid, const uint4* blk, const uint8_t* wblob, QueryBatch& qb,
                       int64_t max_n, int* status, long long wait_limit, cudaStream_t st) {
    auto kern = k_forward_tc<KMAX, FEAT, OPS, WARPDEC, GMAX, THIRD>;
    TcCfg c = cfg;
    c.g_cols = fwd_group_cols<OPS, THIRD>(c);
    const int G = fwd_group_count<OPS, THIRD>(c, GMAX);
    const uint32_t wbytes = (uint32_t)OpsTraits<OPS>::wparts * c.w_bytes;
    size_t smem = fwd_stage_off(wbytes, G) + (size_t)G * fwd_third_bytes<THIRD>(c);
    if (WARPDEC) smem += (size_t)G * kTile * (4 * KMAX + 4) * sizeof(float);
    static std::atomic<uint64_t> attrs{~0ull};
    cudaError_t e = set_smem_attrs(kern, smem, carveout_percent(smem + 1024), attrs);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t t0 = 0;
    for (int i = 0; i < qb.nseg; ++i) {
        qb.seg[i].tile0 = t0;
        t0 += (qb.seg[i].n + kTile - 1) / kTile;
    }
    qb.total_tiles = t0;
    int64_t blocks = qb.n_dev ? (max_n + kTile - 1) / kTile : t0;
    if (blocks > sms) blocks = sms;
    if (blocks < 1) blocks = 1;
    return launch_maybe_pdl(kern, dim3((unsigned)blocks), dim3(kThreads * G), smem, st, blk != nullptr, c,
                            static_cast<const typename OpsTraits<OPS>::GridT*>(grid), blk, wblob, qb, status,
                            wait_limit);
}

// The instance of an operand format for this model: up to eight lobes with
// 2, 4 or any features per level, or sixteen lobes.
template <int OPS>
cudaError_t launch_fwd_ops(const TcCfg& c, const void* grid, const uint4* blk, const uint8_t* wblob, QueryBatch& qb, int64_t max_n,
                           int* status, long long wait_limit, bool warp_decode, cudaStream_t st) {
    if (c.base.K > 8) return launch_fwd<16, 0, OPS>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
    if constexpr (!OpsTraits<OPS>::fp32)
        if (warp_decode) return launch_fwd<8, 0, OPS, true>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
    if constexpr (OPS == kThreeBf16) {
        // FP32 has instances that keep the third part in tensor memory too.
        // 4-feature grids take theirs where its columns suffice for four
        // groups (2^18 queries of a 16-wide network: 44 us, with the part in
        // shared memory 47, before elect_one). 2-feature grids' has three
        // groups with two levels' gathers in flight, against four with one,
        // whose rounds of tiles take about 1.37 times as long: whichever needs
        // less for the rounds of this batch (GB300, 16 levels, 64-wide layers,
        // three and four groups: 3,000 queries 16.5 and 18.5 us; 2^16 40.4 and
        // 36.5; 2^17 63.2 and 60.3; 2^18 97.6 and 109.9; 2^20 343 and 378). The
        // ratio is 1.36 to 1.42 on 16 levels and 1.23 to 1.25 on two to eight, where
        // the rule errs on large batches (2^18 on eight levels: 69.7 and 70.8;
        // 2^20: 237 and 227, two levels 173 and 169). Of the two-part formats
        // three groups gain nothing (FP32 accuracy, 2^20: 320 against 312).
        if (c.base.feat == 4 && 4u * fwd_group_cols<OPS, false>(c) <= 512u)
            return launch_fwd<8, 4, OPS, false, 4, false>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
        if (c.base.feat == 2 && fwd_group_count<OPS, false>(c, 3) == 3) {
            int dev = 0, sms = 1;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            int64_t tiles = 0;
            for (int i = 0; i < qb.nseg; ++i) tiles += (qb.seg[i].n + kTile - 1) / kTile;
            if (qb.n_dev) tiles = (max_n + kTile - 1) / kTile;
            const int64_t r3 = (tiles + 3 * sms - 1) / (3 * sms), r4 = (tiles + 4 * sms - 1) / (4 * sms);
            if (137 * r4 >= 100 * r3)
                return launch_fwd<8, 2, OPS, false, 3, false>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
        }
    }
    if (c.base.feat == 2) return launch_fwd<8, 2, OPS>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
    if (c.base.feat == 4) return launch_fwd<8, 4, OPS>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
    return launch_fwd<8, 0, OPS>(c, grid, blk, wblob, qb, max_n, status, wait_limit, st);
}

}  // namespace tc
}  // namespace npm
