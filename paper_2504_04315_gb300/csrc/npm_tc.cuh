// npm_tc.cuh -- shared pieces of the tensor-core (tcgen05) kernels on
// sm_103a: the model's layer layout for the MMAs and the inline-PTX helpers
// (tensor memory, MMA issue, mbarriers, shared-memory matrix descriptors and
// the BF16 operand stores). Internal to the library.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "npm_device.cuh"

namespace npm {
namespace tc {

constexpr int kTile = 128;
// Operand tiles in shared memory that the kernels write (128 rows x columns,
// 16 bits) are stored in planes of 8 columns: kPlane bytes a plane, 16 bytes
// a row. Core matrices (8 rows x 16 bytes) then lie 128 bytes apart along the
// rows and kPlane along the columns in every tile, whatever its width.
constexpr uint32_t kPlane = kTile * 16;
constexpr int kThreads = 128;

struct TcLayer {
    int K, N;        // logical widths
    int Kp, Np;      // padded to multiples of 16
    uint32_t w_off;  // byte offset of this layer's weights in the blob
    uint32_t idesc;  // instruction descriptor
};

struct TcCfg {
    DevCfg base;
    TcLayer layer[NPM_MAX_LAYERS];
    uint32_t w_bytes;  // bytes of one weight blob (multiple of 128); the
                       // residual (lo) blob follows when split
    int parts, wparts; // 16-bit operand parts of an activation and of a weight
    int split;         // 1: two BF16 parts (three MMAs per K step)
    int f16;           // 1: FP16 operands: activations rounded to FP16, weights
                       // FP16 plus an FP16 residual (two MMAs per K step);
                       // with split, activations FP16 plus an FP16 residual too
    int fp32;          // 1: FP32 or the FP32-accuracy mode (FP32 grid table, the
                       // FP32 path's sampler)
    // Tensor-memory columns of a forward tile group: d_cols of accumulator,
    // then one a_cols wide block per activation part (two 16-bit values to a
    // column; an instance may keep a third part in shared memory instead),
    // g_cols in all (set per launch).
    uint32_t d_cols, a_cols, g_cols;
    // Corner blocks (below): bit l set where level l has them, and the level's
    // first block.
    uint32_t blk_mask;
    uint32_t blk_off[NPM_MAX_LEVELS];
};

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, no swizzle (core matrices of 8 rows x
// 16 bytes): lbo = byte step between core matrices along K, sbo = byte step
// between 8-row groups along M/N; bit 46 is the tcgen05 descriptor version.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// The same with the A operand in tensor memory: lane m holds row m, each
// 32-bit column two consecutive K elements (eight columns per K step of 16).
__device__ __forceinline__ void mma_tmem_a(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// One thread of a converged warp, for the MMAs and their commit. Their operands
// are warp-uniform and computed by the whole warp from uniform values
// (warp_uniform, parameters), and the branch is taken by an elected thread: an
// MMA then issues every 80 cycles or so, against 210-250 under `t == 0`, where
// the operands of each are moved from the thread's registers first. Issue was a
// third of a tile's time (GB300, per tile of the paper-shaped grid, FP32: 12,600
// of 44,500 cycles, now 4,800 of 33,000). A predicate on each instruction, steps
// unrolled in full, or another warp of each group issuing all measured slower
// (2^20 queries: 410, 416 and 382 us against 360).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}\n"
        : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// f(constant) where a layer has 2, 4 or 8 K steps of 16 (32, 64 or 128 values,
// the widths of most networks), else f with 0, for the count at run time: with
// the steps' descriptors as constant offsets an MMA issues in fewer cycles
// (GB300, 2^20 queries, FP32: paper-shaped grid 360 -> 344 us, the paper's own
// 259 -> 239; FP16 235 -> 232, 145 -> 142). Not in the training kernel: 594 ->
// 601 us a step.
template <int N>
struct Steps {
    static constexpr int count = N;
};
template <typename F>
__device__ __forceinline__ void with_steps(int nk, F&& f) {
    if (nk == 4) f(Steps<4>{});
    else if (nk == 2) f(Steps<2>{});
    else if (nk == 8) f(Steps<8>{});
    else f(Steps<0>{});
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// One potentially blocking test of phase `parity`: the thread sleeps in the
// barrier until the phase completes or about 20 microseconds pass (the
// suspend-time hint), so a waiting warp issues almost nothing.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of the barrier; false after ~2^32 cycles.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > (1ll << 32)) return false;
    return true;
}

// Wait bounded by `limit` SM clock cycles (<= 0: one non-blocking test).
__device__ __forceinline__ bool mbar_wait_limit(uint32_t bar, uint32_t parity, long long limit) {
    if (limit <= 0) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.b32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        return ok != 0;
    }
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}

// N consecutive 32-bit columns of this thread's TMEM lane written from
// registers; tmem_wait_st completes the thread's earlier stores.
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[1]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(r[0]) : "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[2]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(taddr), "r"(r[0]), "r"(r[1])
                 : "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[3]) {
    const uint32_t a[2] = {r[0], r[1]}, b[1] = {r[2]};
    tmem_st(taddr, a);
    tmem_st(taddr + 2u, b);
}
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 16 consecutive FP32 columns of this thread's TMEM lane. The values are
// valid only after tmem_wait16 on the same registers.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// tcgen05.wait::ld with the loaded registers as in/out operands, so that no
// use of them can be scheduled before the wait.
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// The same for two columns.
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t (&r)[2]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait2(uint32_t (&r)[2]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]) : : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

// (a, b) rounded to nearest FP16 and packed (a in the low half); values
// beyond the FP16 range saturate to +-65504 rather than becoming infinite.
__device__ __forceinline__ uint32_t pack_f16_sat(float a, float b) {
    uint32_t d;
    asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

// Named barrier of 128-thread tile group g of a CTA (id 1 + g; id 0 is the
// CTA-wide __syncthreads), and its form that also ORs a predicate over the
// group's threads.
__device__ __forceinline__ void tc_group_sync(int g) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(128) : "memory");
}
__device__ __forceinline__ bool tc_group_sync_or(int g, bool p) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred q, o;\n\t"
        "setp.ne.u32 q, %3, 0;\n\t"
        "bar.red.or.pred o, %1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, o;\n\t}\n"
        : "=r"(r)
        : "r"(1 + g), "r"(128), "r"((uint32_t)p)
        : "memory");
    return r != 0;
}

// FP16 residuals (a - hi_a, b - hi_b) of a packed FP16 pair hp = (hi_a,
// hi_b), rounded to nearest and packed the same way.
__device__ __forceinline__ uint32_t f16_residual(uint32_t hp, float a, float b) {
    const float2 hf = __half22float2(*reinterpret_cast<const __half2*>(&hp));
    return pack_f16_sat(a - hf.x, b - hf.y);
}

// Byte offset of element (row, k) in a K-major no-swizzle tile whose rows
// hold kp elements: 8x8 core matrices (128 bytes), K-adjacent core matrices
// 128 bytes apart, 8-row groups kp/8 * 128 bytes apart.
__device__ __forceinline__ uint32_t tile_off(int row, int k, int kp) {
    return (uint32_t)((row >> 3) * (kp >> 3) * 128 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// One or two BF16 values and their residuals lo_off bytes on.
__device__ __forceinline__ void store_pair(uint8_t* sA, uint32_t off, float a, float b, uint32_t lo_off) {
    __nv_bfloat162 hb = __floats2bfloat162_rn(a, b);
    *reinterpret_cast<__nv_bfloat162*>(sA + off) = hb;
    const float2 hf = __bfloat1622float2(hb);
    *reinterpret_cast<uint32_t*>(sA + lo_off + off) = pack_bf16(a - hf.x, b - hf.y);
}

__device__ __forceinline__ void store_one(uint8_t* sA, uint32_t off, float a, uint32_t lo_off) {
    const __nv_bfloat16 hb = __float2bfloat16_rn(a);
    *reinterpret_cast<__nv_bfloat16*>(sA + off) = hb;
    *reinterpret_cast<__nv_bfloat16*>(sA + lo_off + off) = __float2bfloat16_rn(a - __bfloat162float(hb));
}

constexpr float kL2E = 1.4426950408889634f;  // log2(e)
constexpr float kLn2 = 0.69314718055994531f;

// Hardware approximations (PTX ex2/lg2/rcp/sin/cos .approx): e^x is
// evaluated as 2^(x log2 e) with the scaling folded into the caller's FMA.
__device__ __forceinline__ float hw_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// The same where results below 2^-126 count (densities and kappa; 0.1 to 0.3 %
// of a query's time).
__device__ __forceinline__ float hw_ex2_tiny(float x) {
    float y;
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float hw_lg2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float hw_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// Sampler of the reduced-precision path (Sec. 5.3, Jakob's inversion as in
// vmf_sample) on the hardware approximations: 1 - e^{-2k} and log(1 + y) by
// their series where the direct forms lose relative accuracy (2k < 0.1,
// four terms, truncation < 1e-6 relative; |y| < 1/16, seven terms,
// truncation < 1e-9 relative), the fast exponential, logarithm and divide
// elsewhere, and sqrt as x rsqrt(x). The fast logarithm's absolute error
// (about 2^-21.4 near 1) is at most 6e-6 of log(1 + y) for |y| >= 1/16. The
// density is always evaluated at the direction returned, so its accuracy
// bar does not depend on these approximations.
__device__ __forceinline__ void vmf_sample_rp(const Lobe& L, float u1, float u2, float out[3]) {
    const float k = L.kap;
    const float x = 2.0f * k;
    const float em1 = x < 0.1f ? -x * (1.0f - x * (0.5f - x * (1.0f / 6.0f - x * (1.0f / 24.0f))))
                               : __expf(-x) - 1.0f;  // e^{-2k} - 1
    const float y = u1 * em1;                        // in (-1, 0]
    const float ser =
        y * (1.0f + y * (-0.5f + y * (1.0f / 3.0f + y * (-0.25f + y * (0.2f + y * (-1.0f / 6.0f + y * (1.0f / 7.0f)))))));
    const float l1p = fabsf(y) < 0.0625f ? ser : __logf(1.0f + y);
    float t1 = k > 1e-20f ? __fdividef(-l1p, k) : 2.0f * u1;
    t1 = fminf(fmaxf(t1, 0.0f), 2.0f);
    const float W = 1.0f - t1;
    const float q = t1 * (2.0f - t1);
    const float sn = q > 0.0f ? q * rsqrtf(q) : 0.0f;
    float sp, cp;
    __sincosf(2.0f * kPi * (u2 - 0.5f), &sp, &cp);
    const float lx = -sn * cp, ly = -sn * sp;
    float tt[3], bb[3];
    frame(L.mu, tt, bb);
#pragma unroll
    for (int a = 0; a < 3; ++a) out[a] = lx * tt[a] + ly * bb[a] + W * L.mu[a];
}

// ------------------------------------------------------------ grid gathers

// Features 4h .. 4h+3 of entry idx of a table with F = 4 or 8 features: the
// raw 8-byte FP16 or 16-byte FP32 vector, widened to float4 at use.
__device__ __forceinline__ uint2 load_raw4(const __half* g, uint32_t idx, int F, int h) {
    return __ldg(reinterpret_cast<const uint2*>(g) + (size_t)idx * (F >> 2) + h);
}
__device__ __forceinline__ float4 load_raw4(const float* g, uint32_t idx, int F, int h) {
    return __ldg(reinterpret_cast<const float4*>(g) + (size_t)idx * (F >> 2) + h);
}
__device__ __forceinline__ float4 widen4(uint2 raw) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 widen4(float4 v) { return v; }
__device__ __forceinline__ float load_feat(const __half* e, int f) { return __half2float(e[f]); }
__device__ __forceinline__ float load_feat(const float* e, int f) { return __ldg(e + f); }

// Corner blocks: for every entry e of a dense level of 2 or 4 features, the
// 32 bytes that hold the corners a cell with lowest entry e reads together,
// copied from the table: all 8 corners (2 FP16 features), the 4 of a z plane
// (2 FP32 or 4 FP16 features) or the 2 of a row (4 FP32 features), x fastest.
// One 32-byte load then takes the place of 6, 3, 4 or 2 loads on average: the
// L1 serves random gathers one lane a cycle, whatever their width.
__host__ __device__ constexpr int blk_corners(int feat, int value_bytes) { return 32 / (feat * value_bytes); }

struct Block32 {
    uint32_t r[8];
};
// Plain loads, unlike the table's: a forward launched as a dependent of
// k_corner_blocks runs while that still writes the blocks, and reads them
// after its wait (their addresses depend on positions that it reads after it).
__device__ __forceinline__ Block32 load_block(const uint4* blk, uint32_t e) {
    Block32 b;
    asm("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(b.r[0]), "=r"(b.r[1]), "=r"(b.r[2]), "=r"(b.r[3]), "=r"(b.r[4]), "=r"(b.r[5]), "=r"(b.r[6]),
          "=r"(b.r[7])
        : "l"(blk + 2 * (size_t)e));
    return b;
}

// Corner features of one level of 2 features as loaded: nothing here waits
// for the loads, so that several levels' are in flight before the first is
// blended (a select on a loaded value, or a branch around one, would wait).
//
// From the table: a pair of x-neighbours in one load of twice the width where
// they form an aligned pair (half of a level's), else in two.
template <typename GT>
struct Level2;

// The four pairs of x-neighbours of a cell: entries a, b, whether they form an
// aligned pair (then a is its first entry) and whether that comes swapped. On
// a hashed level the neighbours i, i + 1 differ in bit 0 alone exactly when i
// is even, for all four pairs alike; on a dense one they are always adjacent.
struct Pairs {
    uint32_t a[4], b[4], pair[4], swap;
    __device__ __forceinline__ Pairs(const DevCfg& cfg, int l, const Cell& cl) {
        const uint32_t odd = (cfg.level_off[l] + cfg.grid_shift) & 1u;
        swap = 0u;
        if ((cfg.dense_mask >> l) & 1u) {
            const uint32_t D = (uint32_t)cfg.level_res[l];
            const uint32_t e = bounded_index(cl.c[0] + D * (cl.c[1] + D * cl.c[2]), D * D * D - D * D - D - 1u);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = e + ((i & 1) ? D : 0u) + ((i & 2) ? D * D : 0u);
                b[i] = a[i] + 1u;
                pair[i] = (a[i] ^ odd ^ 1u) & 1u;
            }
        } else {
            const uint32_t hy0 = cl.c[1] * 2654435761u, hz0 = cl.c[2] * 805459861u;
            const uint32_t hy[2] = {hy0, hy0 + 2654435761u}, hz[2] = {hz0, hz0 + 805459861u};
            const uint32_t even = (cl.c[0] & 1u) == 0u && odd == 0u ? 1u : 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t h = hy[i & 1] ^ hz[i >> 1];
                const uint32_t e = (cl.c[0] ^ h) & cfg.table_mask;
                b[i] = ((cl.c[0] + 1u) ^ h) & cfg.table_mask;
                swap |= (e & even) << i;
                a[i] = e & ~even;
                pair[i] = even;
            }
        }
    }
};

__device__ __forceinline__ uint32_t corner_idx1(const DevCfg& cfg, int l, const Cell& cl, int c);

template <>
struct Level2<float> {
    float r[16];
    uint32_t swap;  // bit i: pair i swapped
    __device__ __forceinline__ void load_blocks(const uint4* blk, uint32_t e, uint32_t DD) {
        const Block32 b[2] = {load_block(blk, e), load_block(blk, e + DD)};
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = __uint_as_float(b[i >> 3].r[i & 7]);
        swap = 0u;
    }
    __device__ __forceinline__ void load_table(const DevCfg& cfg, const float* __restrict__ table, int l,
                                               const Cell& cl) {
        const float* g = table + (size_t)cfg.level_off[l] * 2;
        const Pairs p(cfg, l, cl);
        swap = p.swap;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm("{\n\t.reg .pred p;\n\t"
                "setp.ne.u32 p, %6, 0;\n\t"
                "@p ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n\t"
                "@!p ld.global.nc.v2.f32 {%0, %1}, [%4];\n\t"
                "@!p ld.global.nc.v2.f32 {%2, %3}, [%5];\n\t}\n"
                : "=f"(r[4 * i]), "=f"(r[4 * i + 1]), "=f"(r[4 * i + 2]), "=f"(r[4 * i + 3])
                : "l"(g + 2 * (size_t)p.a[i]), "l"(g + 2 * (size_t)p.b[i]), "r"(p.pair[i]));
    }
    __device__ __forceinline__ float2 blend(const Cell& cl) const {
        float w[8];
        corner_w8(cl, w);
        float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool sw = (swap >> i) & 1u;
            const float wa = sw ? w[2 * i + 1] : w[2 * i], wb = sw ? w[2 * i] : w[2 * i + 1];
            s.x = fmaf(wa, r[4 * i], s.x);
            s.y = fmaf(wa, r[4 * i + 1], s.y);
            s.x = fmaf(wb, r[4 * i + 2], s.x);
            s.y = fmaf(wb, r[4 * i + 3], s.y);
        }
        return s;
    }
};

template <>
struct Level2<__half> {
    uint32_t r[8];  // corners; from the table pair i may come swapped
    uint32_t swap;
    __device__ __forceinline__ void load_blocks(const uint4* blk, uint32_t e, uint32_t) {
        const Block32 b = load_block(blk, e);
#pragma unroll
        for (int i = 0; i < 8; ++i) r[i] = b.r[i];
        swap = 0u;
    }
    __device__ __forceinline__ void load_table(const DevCfg& cfg, const __half* __restrict__ table, int l,
                                               const Cell& cl) {
        const uint32_t* g = reinterpret_cast<const uint32_t*>(table) + cfg.level_off[l];
        const Pairs p(cfg, l, cl);
        swap = p.swap;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm("{\n\t.reg .pred p;\n\t"
                "setp.ne.u32 p, %4, 0;\n\t"
                "@p ld.global.nc.v2.b32 {%0, %1}, [%2];\n\t"
                "@!p ld.global.nc.b32 %0, [%2];\n\t"
                "@!p ld.global.nc.b32 %1, [%3];\n\t}\n"
                : "=r"(r[2 * i]), "=r"(r[2 * i + 1])
                : "l"(g + p.a[i]), "l"(g + p.b[i]), "r"(p.pair[i]));
    }
    __device__ __forceinline__ float2 blend(const Cell& cl) const {
        float w[8];
        corner_w8(cl, w);
        float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool sw = (swap >> i) & 1u;
            const float wa = sw ? w[2 * i + 1] : w[2 * i], wb = sw ? w[2 * i] : w[2 * i + 1];
            const float2 fa = __half22float2(*reinterpret_cast<const __half2*>(&r[2 * i]));
            const float2 fb = __half22float2(*reinterpret_cast<const __half2*>(&r[2 * i + 1]));
            s.x = fmaf(wa, fa.x, s.x);
            s.y = fmaf(wa, fa.y, s.y);
            s.x = fmaf(wb, fb.x, s.x);
            s.y = fmaf(wb, fb.y, s.y);
        }
        return s;
    }
};

// Corner features of 4 features of a cell with lowest block e; DD = D^2.
__device__ __forceinline__ void gather_blocks4(const uint4* blk, uint32_t e, uint32_t, uint32_t DD,
                                               const __half*, uint2 (&v)[8]) {
    const Block32 b[2] = {load_block(blk, e), load_block(blk, e + DD)};
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = make_uint2(b[c >> 2].r[2 * (c & 3)], b[c >> 2].r[2 * (c & 3) + 1]);
}
__device__ __forceinline__ void gather_blocks4(const uint4* blk, uint32_t e, uint32_t D, uint32_t DD,
                                               const float*, float4 (&v)[8]) {
    const Block32 b[4] = {load_block(blk, e), load_block(blk, e + D), load_block(blk, e + DD),
                          load_block(blk, e + DD + D)};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint32_t* r = &b[c >> 1].r[4 * (c & 1)];
        v[c] = make_float4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
    }
}

// Entry index of corner c of a cell (the corner_idx8 formula for one
// corner; corner 0 is a cell's corner block).
__device__ __forceinline__ uint32_t corner_idx1(const DevCfg& cfg, int l, const Cell& cl, int c) {
    const uint32_t i = cl.c[0] + (c & 1), j = cl.c[1] + ((c >> 1) & 1), k = cl.c[2] + ((c >> 2) & 1);
    if ((cfg.dense_mask >> l) & 1u) {
        const uint32_t D = (uint32_t)cfg.level_res[l];
        return bounded_index(i + D * (j + D * k), D * D * D);
    }
    return (i ^ (j * 2654435761u) ^ (k * 805459861u)) & cfg.table_mask;
}

// ------------------------------------------------------- forward kernels

// Byte offset of the space behind the weights, the barriers and the
// tensor-memory slot of a forward CTA of G tile groups (third activation
// parts; staged raw outputs).
__host__ __device__ inline uint32_t fwd_stage_off(uint32_t wbytes, int G) {
    return (wbytes + 8u * (1u + (uint32_t)G) + 16u + 127u) & ~127u;
}

// The general forward in one operand format (npm_tc_forward.cuh; one
// translation unit per format): grid is the FP16 table, or the FP32 table in
// the formats of FP32 accuracy.
// blk: its corner blocks, or NULL.
template <int OPS>
cudaError_t launch_fwd_ops(const TcCfg& c, const void* grid, const uint4* blk, const uint8_t* wblob, QueryBatch& qb,
                           int64_t max_n, int* status, long long wait_limit, bool warp_decode, cudaStream_t st);

// Operand formats (parts from the highest):
//   kOneBf16   activations and weights rounded to BF16
//   kOneFp16   activations rounded to FP16, weights FP16 plus residual
//   kTwoBf16   activations and weights BF16 plus residual
//   kTwoFp16   activations and weights FP16 plus residual, FP32 grid table
//   kThreeBf16 activations and weights as three BF16 parts (all 24 bits of an
//              FP32 value), FP32 grid table: FP32 arithmetic
enum : int { kOneBf16 = 0, kOneFp16 = 1, kTwoBf16 = 2, kTwoFp16 = 3, kThreeBf16 = 4 };

// Fused forward of the small serving networks (npm_tc_tiny.cu): radiance
// mode, one dense level of 4 features, three layers of at most 32 outputs
// (padded input 16), K = 4, softplus kappa. launch_tiny takes the general
// kernel's configuration, FP16 grid and weight blob. With pdl the kernel is
// launched as a programmatic dependent of the stream's previous kernel: its prologue
// (tensor-memory allocation, copies of the weights and grid) overlaps that
// kernel, which therefore must not write the weights or the grid.
bool tiny_qualifies(const TcCfg& c);
cudaError_t launch_tiny(const TcCfg& c, const __half* grid_h, const uint8_t* wblob, QueryBatch& qb,
                        int64_t max_n, int* status, cudaStream_t st, bool pdl = false);

}  // namespace tc
}  // namespace npm
