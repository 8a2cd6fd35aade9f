// DPQ weight quantizer on the GPU: Algorithm 1 (Sec. 3.1-3.3, Eq. 6-12) with the Cholesky form of
// the update that Sec. 3.3 takes from GPTQ, the least-squared-error search of the group scale,
// and Group-Aware Reordering (Sec. 3.2 and its appendix).
//
// The rows of W are independent; the columns of a row are quantized one after the other, each
// sending its scaled error e to the columns on its right (Eq. 12): w_v <- fma(-e, U_qv, w_v),
// U = upper Cholesky factor of the inverse Hessian in processing order.  Work is cut the way
// GPTQ cuts it, in blocks of one group (128 columns).  Tasks of two kinds: 32 rows of a block are brought up to
// date and quantized (group scale / zero-point, Eq. 8, optional search; the 128 columns in sequence); the errors
// of up to eight blocks are applied to 128 rows of a later column block, q ascending -- the same chain of fused
// multiply-adds, in the same order, that the column-by-column algorithm performs for each element.  One persistent
// launch (dpq_kernel) takes the tasks in an order in which each follows those it waits for.
// Every floating-point step that decides an integer is one explicitly rounded fp32 operation
// (__fmul_rn, __fmaf_rn ...: never contracted; quotients correctly rounded), and the search compares exact integer
// sums, so the codes do not depend on how the work is spread over threads.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "w4a8_common.cuh"
#include "w4a8_dpq_plan.h"
#include "w4a8_ptx.cuh"
#include "w4a8_simple_kernels.cuh"

namespace w4a8 {

// ---- Group-Aware Reordering -----------------------------------------------------------------
// Inside each group the columns go by descending Hessian diagonal, the groups by descending
// maximum diagonal; ties keep the original order.  Ranks are found by counting (exact compares).
__global__ void __launch_bounds__(128)
gar_within_kernel(const float* __restrict__ hdiag, int32_t* __restrict__ within, float* __restrict__ gmax) {
    __shared__ float d[128];
    __shared__ float red[4];
    const int g = blockIdx.x, i = threadIdx.x;
    const float di = hdiag[(int64_t)g * 128 + i];
    d[i] = di;
    __syncthreads();
    int rank = 0;
    for (int j = 0; j < 128; ++j) rank += (d[j] > di || (d[j] == di && j < i)) ? 1 : 0;
    within[(int64_t)g * 128 + rank] = g * 128 + i;
    float m = warp_max(di);
    if ((i & 31) == 0) red[i >> 5] = m;
    __syncthreads();
    if (i == 0) gmax[g] = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
}

__global__ void __launch_bounds__(128)
gar_order_kernel(const int32_t* __restrict__ within, const float* __restrict__ gmax, int G,
                 int32_t* __restrict__ perm) {
    const int g = blockIdx.x;
    const float mg = gmax[g];
    int rank = 0;
    for (int j = 0; j < G; ++j) {
        const float mj = gmax[j];
        rank += (mj > mg || (mj == mg && j < g)) ? 1 : 0;
    }
    perm[(int64_t)rank * 128 + threadIdx.x] = within[(int64_t)g * 128 + threadIdx.x];
}

// work[n][p] = W[n][perm[p]]: the rows in processing order; the marks of dpq_kernel (see DpqMarks); and, once the kernel before has found
// the largest magnitudes, Eq. 6.
__global__ void __launch_bounds__(256)
dpq_gather_kernel(const float* __restrict__ W, const int32_t* __restrict__ perm, int64_t N, int64_t K,
                  float* __restrict__ work, uint8_t* __restrict__ codes, uint16_t* __restrict__ gscale, float* s_w, int64_t scales) {
    ptx::griddep_launch_dependents();
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= N * K) return;
    const int64_t n = i / K, p = i - n * K;
    work[i] = W[n * K + (perm ? perm[p] : (int32_t)p)];
    if (n % 32 == 0 && (p & 127) == 0) {   // (the first row's hold control words too)
        uint4* c = reinterpret_cast<uint4*>(codes + n * (K >> 1) + (p >> 1));
        c[0] = c[3] = make_uint4(0u, 0u, 0u, 0u);
        gscale[n * (K >> 7) + (p >> 7)] = 0xFFFFu;
    }
    if (i < scales) {
        ptx::griddep_wait();
        amax_to_scale(s_w + i);
    }
}

// ---- Eq. 8 / Eq. 9 / Eq. 10 on one FP8-valued weight ------------------------------------------
struct DpqGroup {
    float s;  // group scale (a BF16 value)
    int z;    // zero-point
};

__device__ __forceinline__ DpqGroup dpq_group_params(float lo, float hi, float amax, float p, int symmetric) {
    DpqGroup g;
    if (symmetric) {
        const float a = __fmul_rn(p, amax);
        g.s = (a > 0.0f) ? __fdiv_rn(a, 7.0f) : 1.0f;
        g.z = 8;
        g.s = __bfloat162float(__float2bfloat16_rn(g.s));
    } else {
        const float l = __fmul_rn(p, lo), h = __fmul_rn(p, hi);
        g.s = (h > l) ? __fdiv_rn(__fsub_rn(h, l), 15.0f) : 1.0f;  // Eq. 8
        g.s = __bfloat162float(__float2bfloat16_rn(g.s));
        const float zf = rintf(__fdiv_rn(-l, g.s));
        g.z = (int)fminf(fmaxf(zf, 0.0f), 15.0f);
    }
    return g;
}

// ---- division by a repeated divisor --------------------------------------------------------------
// The correctly rounded quotient from the reciprocal h = RN(1 / b) and its tail l, in four dependent
// operations: q = RN(a h + RN(a l)) is within half a unit in the last place and 2^-24 of a / b, its remainder is exact
// in one FMA, and the correction by the remainder times a correctly rounded reciprocal then rounds to
// RN(a / b) (Markstein's theorem, IBM J. Res. Dev. 34(1), 1990).  Valid while nothing underflows or
// overflows on the way: |b| in [2^-40, 2^40], a = 0 or |a| in [2^-72, 2^60]; a zero quotient may lose its sign.
struct Recip {
    float b, h, l;
};
__device__ __forceinline__ Recip make_recip(float b) {
    Recip r;
    r.b = b;
    r.h = __fdiv_rn(1.0f, b);
    r.l = __fmul_rn(__fmaf_rn(-r.h, b, 1.0f), r.h);
    return r;
}
__device__ __forceinline__ float div_recip(float a, const Recip& r) {
    const float q = __fmaf_rn(a, r.h, __fmul_rn(a, r.l));
    return __fmaf_rn(__fmaf_rn(-q, r.b, a), r.h, q);
}
__device__ __forceinline__ bool recip_range(float b) { return fabsf(b) >= 0x1p-40f && fabsf(b) <= 0x1p40f; }

// Two FP32 operations in one instruction (each rounded once, as two scalar ones).
__device__ __forceinline__ unsigned long long div_recip_f32x2(unsigned long long a, const Recip& r) {
    const unsigned long long h = pack_f32x2(r.h, r.h);
    const unsigned long long q = fma_f32x2(a, h, mul_f32x2(a, pack_f32x2(r.l, r.l)));
    return fma_f32x2(fma_f32x2(q, pack_f32x2(-r.b, -r.b), a), h, q);
}

// 16 bytes (four floats) global -> shared, asynchronously; four 4-byte copies where the source is not
// 16-byte aligned.
__device__ __forceinline__ void dpq_copy16(uint32_t dst, const float* src, bool vec) {
    if (vec) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * i), "l"(src + i) : "memory");
    }
}
__device__ __forceinline__ void dpq_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void dpq_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// nearest_Z of two values (Eq. 10), through the conversion instructions.
__device__ __forceinline__ float2 e4m3x2_roundtrip(float a, float b) {
    uint32_t h2;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)cvt_e4m3x2(b, a)));
    return __half22float2(*reinterpret_cast<const __half2*>(&h2));
}

// Four columns of the chain with IEEE divisions, for operands outside the range of div_recip: v[0..3] the weights,
// v[4..7] receives their errors (negated), u_d the block of U from (q0, q0) on; returns the four FP8 codes.
__device__ __noinline__ uint32_t dpq_four_slow(float* v, float sw, const float* lut_h, const float* u_d) {
    uint32_t all = 0;
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        const uint32_t code = cvt_e4m3x2(0.0f, __fdiv_rn(v[c], sw));
        v[4 + c] = __fdiv_rn(__fsub_rn(lut_h[code], v[c]), u_d[c * 128 + c]);
        for (int j = c + 1; j < 4; ++j) v[j] = __fmaf_rn(v[4 + c], u_d[c * 128 + j], v[j]);
        all |= code << (8 * c);
    }
    return all;
}

template <int W>   // lanes that share a row
__device__ __forceinline__ float row_min(float v) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
template <int W>
__device__ __forceinline__ float row_max(float v) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
template <int W>
__device__ __forceinline__ long long row_sum_ll(long long v) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Progress is marked in the outputs, where these are not written yet, so that a call needs no memory beside its work array:
//   * gscale of the first of 32 rows and a block: 0xFFFF until the block's errors for those rows are in place (no scale has these
//     bits: a NaN is rounded to 0x7FFF);
//   * the last word of that row's codes of a column block: how many blocks' errors its 32 rows have taken (of no use, and
//     overwritten with codes, once the block itself is done);
//   * the word before it: not 0 once the block's first 96 columns are done, whose errors the next block's task can take
//     beside the rest of the chain (and of no use when the block is done);
//   * the first words of the first row's codes of the last block: tickets handed out, CTAs that have left, abort.  What belongs
//     there waits in the work array until the last CTA leaves.
struct DpqMarks {
    uint8_t* codes;
    uint16_t* gscale;
    const int32_t* perm;
    int64_t K;
    __device__ __forceinline__ int64_t group(int b) const { return perm ? (int64_t)(__ldg(perm + (int64_t)b * 128) >> 7) : (int64_t)b; }
    __device__ __forceinline__ uint16_t* done(int64_t rows32, int b) const { return gscale + rows32 * 32 * (K >> 7) + group(b); }
    __device__ __forceinline__ unsigned int* applied(int64_t rows32, int c) const {
        return reinterpret_cast<unsigned int*>(codes + rows32 * 32 * (K >> 1) + group(c) * 64 + 60);
    }
    __device__ __forceinline__ unsigned int* early(int64_t rows32, int b) const { return applied(rows32, b) - 1; }
    __device__ __forceinline__ unsigned int* control() const { return reinterpret_cast<unsigned int*>(codes + group((int)(K >> 7) - 1) * 64); }
};
struct DpqWait {   // bounded polls by single threads
    unsigned int* control;
    unsigned int* status_word;
    template <class Test>
    __device__ __forceinline__ bool until(Test test) const {
        uint64_t t0 = 0;
        uint32_t spins = 0;
        while (!test()) {
            if (spins > 32u) __nanosleep(64);
            if ((++spins & 15u) == 0u) {
                if (*reinterpret_cast<volatile unsigned int*>(control + 2)) return false;
                const uint64_t now = ptx::globaltimer_ns();
                if (t0 == 0) {
                    t0 = now;
                } else if (now - t0 > ptx::kWaitLimitNs) {
                    atomicExch(control + 2, 1u);
                    atomicOr(status_word, kStatusTimeout);
                    return false;
                }
            }
        }
        return true;
    }
};
// A copy that is still on its way when a CTA gives up.
__device__ __forceinline__ void dpq_land(uint32_t bar, uint32_t parity) {
    const uint64_t t0 = ptx::globaltimer_ns();
    while (!ptx::mbar_try_wait(bar, parity) && ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs / 20) {
    }
}
struct DpqMaps {
    CUtensorMap u;        // U [K][K], box 128 x 32 (only used where U is 16-byte aligned)
    CUtensorMap errors;   // the work array as [N / 4][4][K], box 128 x 1 x 32: where errors are kept, see dpq_load_errors
};
__device__ __forceinline__ uint16_t dpq_ld_acquire_u16(const uint16_t* p) {
    uint16_t v;
    asm volatile("ld.acquire.gpu.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return v;
}
constexpr int kDpqThreads = 256;
constexpr int kDpqRowsPerCta = 32;      // eight lanes per row
constexpr int kDpqChunk = 32;           // values of q per stage
struct DpqSmem {
    // block CTAs
    static constexpr int kU = 0;                                   // [128][128] U of the block itself
    static constexpr int kPanel = kU + 128 * 128 * 4;              // 2 x [32][128] U of the previous block's rows
    static constexpr int kErr = kPanel + 2 * kDpqChunk * 128 * 4;  // 2 x [32][32 rows] errors of the previous block
    static constexpr int kCodes = kErr + 2 * kDpqChunk * kDpqRowsPerCta * 4 + 256;
    static constexpr int kDiag = kCodes + kDpqRowsPerCta * 128;    // [128] float4: U_qq, its reciprocal and tail
    static constexpr int kPerm = kDiag + 128 * 16;                 // [128] column within its original group
    static constexpr int kBlockBytes = kPerm + 128 + 16;
    // over the panel and the errors, idle by then: the rows' tables
    static constexpr int kLutPitch = 257;                          // floats; rows a bank apart
    static constexpr int kLut = kPanel;
    static constexpr int kLutU = kLut + kDpqRowsPerCta * kLutPitch * 4;
    static_assert(kLutU + kDpqRowsPerCta * 256 <= kCodes, "tables");
    // applications: a stage is 32 q of U [32][128] and of the errors [32 groups of four rows][32 q][4]
    static constexpr int kStages = 3;
    static constexpr int kStageU = kDpqChunk * 128 * 4;
    static constexpr int kStage = 2 * kStageU;
    static constexpr int kTrailBytes = kStages * kStage;
    static constexpr int kBytes = kBlockBytes > kTrailBytes ? kBlockBytes : kTrailBytes;
    static_assert(2 * (kBytes + 1024) <= 228 * 1024, "two CTAs per SM");
};

// Where the (negated) errors of a block are kept: in place of the block's weights, which nothing reads any
// more, and in the order in which they are wanted, four rows of one q side by side: row 4 g + j of a complete
// group of four rows holds q = 32 j .. 32 j + 31 as float4 (rows 4 g .. 4 g + 3).  The up to three rows after the last
// complete group keep their own errors, q ascending.
//
// Chunk c (32 values of q) of the rows from n0 on -> e_s[q][ROWS], the groups of row q permuted by ^ (q & 7) so that the
// copies (consecutive q) fall into different banks.
template <int ROWS>
__device__ __forceinline__ void dpq_load_errors(float* e_s, uint32_t e_addr, const float* __restrict__ work, int64_t N,
                                                int64_t K, int64_t p, int64_t n0, int c) {
    const int q = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < ROWS / 4 * 32 / kDpqThreads; ++i) {
        const int g = (int)(threadIdx.x >> 5) + i * (kDpqThreads / 32);
        const int64_t n = n0 + 4 * g;
        const int at = q * ROWS + 4 * (g ^ (q & 7));
        if (n + 3 < N) {
            dpq_copy16(e_addr + (uint32_t)at * 4u, work + (n + c) * K + p + 4 * q, true);
        } else {
#pragma unroll
            for (int r = 0; r < 4; ++r) e_s[at + r] = n + r < N ? __ldcg(work + (n + r) * K + p + c * kDpqChunk + q) : 0.0f;
        }
    }
}

// Columns further to the right, w[n][v] <- fma(-e[n][q], U[q][v], w[n][v]) for the q of one block or of two in
// ascending order: the chain of fused multiply-adds that the column-by-column algorithm performs for that element.
// 128 rows x 128 columns per CTA; a warp takes 16 rows and all columns, a lane four columns.  Bound: the FP32 pipes,
// if shared memory keeps up: per q a warp reads 512 distinct bytes of U and sixteen errors that all lanes share
// (five 16-byte loads, eight 128-byte passes), half of what an 8 x 8 tile per thread takes, whose lanes read the
// same words from different quarters of the warp; the operands of the next q are fetched ahead (waiting for them
// was the largest stall with four warps per scheduler).  Packed pairs of rows: the pipe takes a packed FMA every other
// cycle, which leaves issue slots for the loads; this loop on its own runs at 30 T FMA/s (16 x 8 per thread and one CTA per
// SM: 32; operands that are repeated in shared memory instead of registers: 25-27).  Errors and rows of U come by tile loads,
// 32 q a stage, two stages ahead.
__device__ __forceinline__ bool dpq_trailing_tile(uint8_t* sm, uint32_t sm_addr, float* work, const float* __restrict__ U,
                                                  int64_t N, int64_t K, int e0, int blocks, int col, int64_t n0, bool uvec,
                                                  const DpqMarks& marks, const DpqWait& wait, const DpqMaps& maps, uint32_t bars,
                                                  volatile uint32_t* abort_s, uint32_t& ring) {
    const int64_t pprev = (int64_t)e0 * 128, v0 = (int64_t)col * 128;
    constexpr int kPerBlock = 128 / kDpqChunk;
    const int chunks = blocks * kPerBlock;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int groups = (int)(N - n0 >= 128 ? 32 : (N - n0) >> 2);   // complete groups of four rows
    const bool tail = groups < 32 && n0 + 4 * groups < N;           // up to three rows behind the last one
    // Stage of chunk c, counted over all tasks in `ring`: one tile load for 32 rows of U, one for the errors of 32 groups.
    auto stage = [&](int c) { return (int)((ring + (uint32_t)c) % DpqSmem::kStages); };
    auto parity = [&](int c) { return ((ring + (uint32_t)c) / DpqSmem::kStages) & 1u; };
    auto load_u = [&](int c) {
        const uint32_t dst = sm_addr + (uint32_t)(stage(c) * DpqSmem::kStage), bar = bars + 8u * (uint32_t)stage(c);
        const int q = (int)pprev + c * kDpqChunk;
        if (warp == 0 && ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx(bar, (uint32_t)(uvec ? DpqSmem::kStage : DpqSmem::kStageU));
            if (uvec) ptx::tma_load_2d(dst, &maps.u, (int)v0, q, bar);
        }
        if (!uvec) {
#pragma unroll
            for (int i = 0; i < kDpqChunk / 8; ++i)
                dpq_copy16(dst + (uint32_t)(i * 8 * 512 + tid * 16), U + (int64_t)(q + 8 * i + warp) * K + v0 + 4 * lane, false);
            dpq_commit();
        }
    };
    auto load_e = [&](int c) {
        const uint32_t dst = sm_addr + (uint32_t)(stage(c) * DpqSmem::kStage + DpqSmem::kStageU), bar = bars + 8u * (uint32_t)stage(c);
        const int x = (int)pprev + (c / kPerBlock) * 128, y = c % kPerBlock, z = (int)(n0 >> 2);
        if (warp == 0 && ptx::elect_one()) ptx::tma_load_3d(dst, &maps.errors, x, y, z, bar);
    };
    // (the marks' addresses come from perm: looked up while U, which is the caller's, is requested)
    const int64_t r32 = n0 / 32 + (tid & 3);
    const uint16_t* done = nullptr;
    const unsigned int* applied = nullptr;
    if (tid < 4 && r32 * 32 < N) done = marks.done(r32, e0 + blocks - 1);
    if (tid == 32 && e0 > 0) applied = marks.applied(n0 / 32, col);
    load_u(0);
    load_u(1);
    {   // the errors of these rows are there, and those before them have been applied to this tile
        bool ok = true;
        if (done) ok = wait.until([&] { return dpq_ld_acquire_u16(done) != 0xFFFFu; });
        else if (applied) ok = wait.until([&] { return ptx::ld_acquire_gpu(applied) >= (unsigned)e0; });
        if (!__syncthreads_and(ok)) {   // given up: what is on its way lands first
            load_e(0);
            load_e(1);
            asm volatile("cp.async.wait_all;" ::: "memory");
            dpq_land(bars + 8u * (uint32_t)stage(0), parity(0));
            dpq_land(bars + 8u * (uint32_t)stage(1), parity(1));
            return false;
        }
    }
    // (what was seen of the other CTAs' writes holds for the tile loads too)
    asm volatile("fence.proxy.async.global;" ::: "memory");
    load_e(0);
    load_e(1);
    float* wp = work + (n0 + 16 * warp) * K + v0 + 4 * lane;
    const int rows = (int)min((int64_t)16, N - (n0 + 16 * warp));   // (may be negative: a warp without rows)
    unsigned long long acc[8][4];   // rows 2 i and 2 i + 1, four columns
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
        if (2 * i < rows) a = __ldcg(reinterpret_cast<const float4*>(wp + (int64_t)(2 * i) * K));
        if (2 * i + 1 < rows) b = __ldcg(reinterpret_cast<const float4*>(wp + (int64_t)(2 * i + 1) * K));
        acc[i][0] = pack_f32x2(a.x, b.x);
        acc[i][1] = pack_f32x2(a.y, b.y);
        acc[i][2] = pack_f32x2(a.z, b.z);
        acc[i][3] = pack_f32x2(a.w, b.w);
    }
#pragma unroll 1
    for (int c = 0; c < chunks; ++c) {
        if (!uvec) {
            if (c + 1 < chunks) dpq_wait<1>();
            else dpq_wait<0>();
        }
        const bool ok = ptx::mbar_wait(bars + 8u * (uint32_t)stage(c), parity(c), abort_s, wait.status_word);
        if (!__syncthreads_and(ok)) {   // chunk c is there; chunk c - 1 has been consumed by everybody
            if (c + 1 < chunks) dpq_land(bars + 8u * (uint32_t)stage(c + 1), parity(c + 1));
            return false;
        }
        if (c + 2 < chunks) {
            load_u(c + 2);
            load_e(c + 2);
        }
        if (tail) {   // (the tile load has put zeros there)
            if (warp == 0) {
                float* e = reinterpret_cast<float*>(sm + stage(c) * DpqSmem::kStage + DpqSmem::kStageU) + groups * 128 + 4 * lane;
                for (int64_t n = n0 + 4 * groups; n < N; ++n)
                    e[n & 3] = __ldcg(work + n * K + pprev + c * kDpqChunk + lane);
            }
            __syncthreads();
        }
        const uint8_t* us = sm + stage(c) * DpqSmem::kStage + 16 * lane;
        const uint8_t* es = sm + stage(c) * DpqSmem::kStage + DpqSmem::kStageU + 4 * warp * 512;
        struct Q {
            ulonglong2 e[4];
            float4 u;
        } q0, q1;
        auto fetch = [&](Q& t, int q8, int j) {   // q = q8 + j, j = 0..7 known at compile time
            t.u = *reinterpret_cast<const float4*>(us + (q8 + j) * 512);
#pragma unroll
            for (int g = 0; g < 4; ++g) t.e[g] = *reinterpret_cast<const ulonglong2*>(es + g * 512 + (q8 + j) * 16);
        };
        auto apply = [&](const Q& t) {
            const float uv[4] = {t.u.x, t.u.y, t.u.z, t.u.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned long long u2 = pack_f32x2(uv[j], uv[j]);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    acc[2 * g][j] = fma_f32x2(t.e[g].x, u2, acc[2 * g][j]);   // Eq. 12
                    acc[2 * g + 1][j] = fma_f32x2(t.e[g].y, u2, acc[2 * g + 1][j]);
                }
            }
        };
        fetch(q0, 0, 0);
#pragma unroll 1
        for (int q8 = 0; q8 < kDpqChunk; q8 += 8) {
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                fetch(q1, q8, j + 1);
                apply(q0);
                if (j < 6) fetch(q0, q8, j + 2);
                else fetch(q0, (q8 + 8) & (kDpqChunk - 1), 0);   // (the last one is not used)
                apply(q1);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float4 a, b;
        unpack_f32x2(acc[i][0], a.x, b.x);
        unpack_f32x2(acc[i][1], a.y, b.y);
        unpack_f32x2(acc[i][2], a.z, b.z);
        unpack_f32x2(acc[i][3], a.w, b.w);
        if (2 * i < rows) *reinterpret_cast<float4*>(wp + (int64_t)(2 * i) * K) = a;
        if (2 * i + 1 < rows) *reinterpret_cast<float4*>(wp + (int64_t)(2 * i + 1) * K) = b;
    }
    ring += (uint32_t)chunks;
    __syncthreads();
    if (tid < 4 && n0 + 32 * tid < N) {
        __threadfence();
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(marks.applied(n0 / 32 + tid, col)), "r"((uint32_t)(e0 + blocks)) : "memory");
    }
    return true;
}

// Block b of 32 rows, eight lanes per row.  Lane sl of a row keeps columns 32 k + 4 sl + {0..3}, k = 0..3.
// Bound by the latency of the column chain (two quotients, a conversion and a look-up each).
// Four columns at a time: every lane of the row fetches the four weights (one exchange per four columns
// instead of one per column), follows the same scalar computation through all four, and then applies
// the four errors to its own columns, in ascending order.  Columns that are finished are updated along
// with the others; nothing reads them again.
__device__ __forceinline__ bool dpq_block_rows(uint8_t* sm, uint32_t sm_addr, float* work, const float* __restrict__ U,
                                               const int32_t* __restrict__ perm, int64_t N, int64_t K, int b, int64_t rows32,
                                               int symmetric, int mse_steps, int per_channel, const float* __restrict__ s_w,
                                               uint8_t* codes, uint16_t* gscale, uint8_t* __restrict__ gzero, bool uvec,
                                               const DpqMarks& marks, const DpqWait& wait) {
    const int64_t p0 = (int64_t)b * 128;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, sl = lane & 7;
    const float* u_s = reinterpret_cast<const float*>(sm + DpqSmem::kU);
    uint8_t* code_s = sm + DpqSmem::kCodes;
    float4* diag_s = reinterpret_cast<float4*>(sm + DpqSmem::kDiag);
    uint8_t* perm_s = sm + DpqSmem::kPerm;
    const int rl = 4 * warp + (lane >> 3);                        // row within the CTA
    const int64_t n_raw = rows32 * kDpqRowsPerCta + rl;
    const bool valid = n_raw < N;                                 // (lanes without a row repeat the last one and store nothing)
    const int64_t n = valid ? n_raw : N - 1;
    const int64_t G = K >> 7;

    auto load_panel = [&](int c) {
        const uint32_t dst = sm_addr + DpqSmem::kPanel + (uint32_t)((c & 1) * kDpqChunk * 128 * 4);
        const float* src = U + (p0 - 128 + c * kDpqChunk) * K + p0;
#pragma unroll
        for (int i = 0; i < kDpqChunk * 32 / kDpqThreads; ++i) {
            const int idx = i * kDpqThreads + tid, q = idx >> 5, c4 = (idx & 31) * 4;
            dpq_copy16(dst + (uint32_t)((q * 128 + c4) * 4), src + (int64_t)q * K + c4, uvec);
        }
    };
    auto load_err = [&](int c) {
        const int off = DpqSmem::kErr + (c & 1) * kDpqChunk * kDpqRowsPerCta * 4;
        dpq_load_errors<kDpqRowsPerCta>(reinterpret_cast<float*>(sm + off), sm_addr + (uint32_t)off, work, N, K, p0 - 128,
                                        rows32 * kDpqRowsPerCta, c);
    };
    // U is the caller's: what is wanted of it first is requested ahead of the wait
    if (b > 0) {
        load_panel(0);
        load_panel(1);
    }
#pragma unroll
    for (int i = 0; i < 128 * 32 / kDpqThreads; ++i) {
        const int idx = i * kDpqThreads + tid, q = idx >> 5, c4 = (idx & 31) * 4;
        dpq_copy16(sm_addr + DpqSmem::kU + (uint32_t)((q * 128 + c4) * 4), U + (p0 + q) * K + p0 + c4, uvec);
    }
    if (tid < 128) perm_s[tid] = (uint8_t)(perm ? (perm[p0 + tid] & 127) : tid);
    if (b == 0) {
        dpq_commit();
    } else {
        // the block before is done but for its last 32 columns, and the errors before its have been applied to this one
        bool ok = true;
        if (tid == 0) {
            const uint16_t* d = marks.done(rows32, b - 1);
            const unsigned int* early = marks.early(rows32, b - 1);
            ok = wait.until([&] { return ptx::ld_acquire_gpu(early) != 0u || dpq_ld_acquire_u16(d) != 0xFFFFu; });
        } else if (tid == 32 && b > 1) {
            const unsigned int* d = marks.applied(rows32, b);
            ok = wait.until([&] { return ptx::ld_acquire_gpu(d) >= (unsigned)(b - 1); });
        }
        if (!__syncthreads_and(ok)) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            return false;
        }
        load_err(0);
        dpq_commit();
        load_err(1);
        dpq_commit();
    }
    // The errors of the previous block first (the tasks that apply errors leave those to the block's own): a
    // warp takes its four rows, a lane four consecutive columns of each, so that U is read once per four rows.
    {
        const int64_t r0 = rows32 * kDpqRowsPerCta + 4 * warp;
        float a[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float4 t = __ldcg(reinterpret_cast<const float4*>(work + (r0 + r < N ? r0 + r : N - 1) * K + p0 + 4 * lane));
            a[r][0] = t.x;
            a[r][1] = t.y;
            a[r][2] = t.z;
            a[r][3] = t.w;
        }
        if (b > 0) {
#pragma unroll 1
            for (int c = 0; c < 128 / kDpqChunk; ++c) {
                // groups in flight, in order: chunk 0 (and all that was requested ahead of the wait), chunk 1, chunk 2, U of chunk 3,
                // errors of chunk 3
                if (c < 3) dpq_wait<1>();
                else dpq_wait<0>();
                __syncthreads();
                const float* us = reinterpret_cast<const float*>(sm + DpqSmem::kPanel) + (c & 1) * kDpqChunk * 128 + 4 * lane;
                const float* es = reinterpret_cast<const float*>(sm + DpqSmem::kErr) + (c & 1) * kDpqChunk * kDpqRowsPerCta;
#pragma unroll 8
                for (int q = 0; q < kDpqChunk; ++q) {
                    const float4 e4 = *reinterpret_cast<const float4*>(es + q * kDpqRowsPerCta + 4 * (warp ^ (q & 7)));
                    const float4 u4 = *reinterpret_cast<const float4*>(us + q * 128);
                    const float ev[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        a[r][0] = __fmaf_rn(ev[r], u4.x, a[r][0]);
                        a[r][1] = __fmaf_rn(ev[r], u4.y, a[r][1]);
                        a[r][2] = __fmaf_rn(ev[r], u4.z, a[r][2]);
                        a[r][3] = __fmaf_rn(ev[r], u4.w, a[r][3]);
                    }
                }
                bool ok = true;
                if (c == 2 && tid == 0) {   // the last 32 columns of the block before
                    const uint16_t* d = marks.done(rows32, b - 1);
                    ok = wait.until([&] { return dpq_ld_acquire_u16(d) != 0xFFFFu; });
                }
                if (!__syncthreads_and(ok)) {
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    return false;
                }
                if (c < 2) load_panel(c + 2);
                if (c == 0 || c == 2) load_err(c == 0 ? 2 : 3);
                dpq_commit();
            }
        } else {
            dpq_wait<0>();
            __syncthreads();
        }
        // to eight lanes per row through the (idle) panel buffers
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *reinterpret_cast<float4*>(sm + DpqSmem::kPanel + ((4 * warp + r) * 132 + 4 * lane) * 4) =
                make_float4(a[r][0], a[r][1], a[r][2], a[r][3]);
        __syncwarp();
    }
    unsigned long long w[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(sm + DpqSmem::kPanel + (rl * 132 + 32 * k + 4 * sl) * 4);
        w[2 * k] = t.x;
        w[2 * k + 1] = t.y;
    }
    if (tid < 128) {
        const float d = u_s[tid * 128 + tid];
        const Recip r = make_recip(d);
        diag_s[tid] = make_float4(d, r.h, r.l, 0.0f);
    }
    const bool diag_ok = __syncthreads_and(tid >= 128 || recip_range(u_s[(tid & 127) * 129]));

    // Eq. 7 on the group's current weights, then Eq. 8 (once per group)
    const Recip sw = make_recip(per_channel ? s_w[n] : s_w[0]);
    float w8[16];
    float lo = 0.0f, hi = 0.0f, amax = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        unpack_f32x2(w[i], w8[2 * i], w8[2 * i + 1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float& v = w8[2 * i + h];
            v = e4m3_roundtrip(__fdiv_rn(v, sw.b));
            lo = fminf(lo, v);
            hi = fmaxf(hi, v);
            amax = fmaxf(amax, fabsf(v));
        }
    }
    lo = row_min<8>(lo);
    hi = row_max<8>(hi);
    amax = row_max<8>(amax);
    DpqGroup grp = dpq_group_params(lo, hi, amax, 1.0f, symmetric);
    // whole-number bounds of u - z + fz: codes 0..15 with the zero-point added, or -7..7 around zero
    const float dlo = symmetric ? -7.0f : 0.0f, dhi = symmetric ? 7.0f : 15.0f;
    if (mse_steps > 1) {
        // Sec. 3.3: least squared error over the group among shrunk ranges; exact integer sums
        long long best = -1;
#pragma unroll 1
        for (int t = 0; t < mse_steps; ++t) {
            const float pt = __fsub_rn(1.0f, __fmul_rn((float)t, 0.02f));
            const DpqGroup gt = dpq_group_params(lo, hi, amax, pt, symmetric);
            const Recip st = make_recip(gt.s);   // (a sixteenth of FP8 values apart: always within the range of div_recip)
            const float fz = symmetric ? 0.0f : (float)gt.z;
            long long e2 = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                // two weights per instruction where there is a packed form
                const unsigned long long v = pack_f32x2(w8[2 * i], w8[2 * i + 1]);
                float c0, c1;
                unpack_f32x2(add_f32x2(div_recip_f32x2(v, st), pack_f32x2(fz, fz)), c0, c1);
                const unsigned long long magic = pack_f32x2(12582912.0f, 12582912.0f);
                unsigned long long d = add_f32x2(pack_f32x2(fminf(fmaxf(c0, dlo), dhi), fminf(fmaxf(c1, dlo), dhi)), magic);
                d = add_f32x2(add_f32x2(d, pack_f32x2(-12582912.0f, -12582912.0f)), pack_f32x2(-fz, -fz));   // u - z
                float p0s, p1s;
                unpack_f32x2(mul_f32x2(d, pack_f32x2(gt.s, gt.s)), p0s, p1s);
                const float2 h8 = e4m3x2_roundtrip(p0s, p1s);
                // 512 (w8 - h8), a whole number below 2^20: both are on the 2^-9 grid
                const unsigned long long diff = add_f32x2(v, pack_f32x2(-h8.x, -h8.y));
                float i0, i1;
                unpack_f32x2(fma_f32x2(diff, pack_f32x2(512.0f, 512.0f), magic), i0, i1);
                const int da = __float_as_int(i0) - 0x4B400000, db = __float_as_int(i1) - 0x4B400000;
                e2 += (long long)da * da;
                e2 += (long long)db * db;
            }
            e2 = row_sum_ll<8>(e2);
            if (best < 0 || e2 < best) {
                best = e2;
                grp = gt;
            }
        }
    }

    const int64_t og = perm ? (int64_t)(perm[p0] >> 7) : (int64_t)b;
    const float fz = symmetric ? 0.0f : (float)grp.z;
    const float uoff = symmetric ? 8.0f : (float)grp.z;
    // The row's table: code and dequantized value (Eq. 9, 10, 11) of each of the 256 FP8 values that Eq. 7 can give.
    // Worked out once per group, off the chain: a column then takes one conversion and one look-up instead of a
    // quotient, two roundings and a product.
    float* lut_h = reinterpret_cast<float*>(sm + DpqSmem::kLut) + rl * DpqSmem::kLutPitch;
    uint8_t* lut_u = sm + DpqSmem::kLutU + rl * 256;
    {
        const Recip sg = make_recip(grp.s);
#pragma unroll 4
        for (int i = 0; i < 16; ++i) {
            const int code = 16 * i + 2 * sl;   // this lane: code and code + 1
            uint32_t h2;
            asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)(code | (code + 1) << 8)));
            const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&h2));
            float d[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float c = fminf(fmaxf(__fadd_rn(div_recip(h == 0 ? v.x : v.y, sg), fz), dlo), dhi);
                d[h] = __fsub_rn(__fsub_rn(__fadd_rn(c, 12582912.0f), 12582912.0f), fz);
            }
            const float2 h8 = e4m3x2_roundtrip(__fmul_rn(d[0], grp.s), __fmul_rn(d[1], grp.s));
            lut_h[code] = __fmul_rn(h8.x, sw.b);
            lut_h[code + 1] = __fmul_rn(h8.y, sw.b);
            *reinterpret_cast<uint16_t*>(lut_u + code) =
                (uint16_t)(__float2int_rn(__fadd_rn(d[0], uoff)) | __float2int_rn(__fadd_rn(d[1], uoff)) << 8);
        }
        __syncwarp();
    }
    // the divisions take the short form where operands are within its range (a weight of zero is)
    // where this row's errors go (see dpq_load_errors): value (row, q) of a complete group of four rows to row 4 g + q / 32
    const bool whole = (n_raw | 3) < N;
    float* ew = whole ? work + (n & ~(int64_t)3) * K + p0 + (n & 3) : work + n * K + p0;
    const bool fast = diag_ok && recip_range(sw.b);
    const float wmin = fast ? 0x1p-40f : __int_as_float(0x7F800000), wzero = fast ? 0.0f : -1.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll 1
        for (int o = 0; o < 8; ++o) {
            const int q0 = 32 * k + 4 * o;
            const float* urow = u_s + q0 * 128;
            float wv[4], ne[4];
            uint32_t code[4];   // Eq. 7, as an FP8 byte
            unpack_f32x2(w[2 * k], wv[0], wv[1]);
            unpack_f32x2(w[2 * k + 1], wv[2], wv[3]);
#pragma unroll
            for (int c = 0; c < 4; ++c) wv[c] = __shfl_sync(0xFFFFFFFFu, wv[c], (lane & 24) | o);
            const float4 u0 = *reinterpret_cast<const float4*>(urow + q0);
            const float4 u1 = *reinterpret_cast<const float4*>(urow + 128 + q0);
            const float u23 = urow[256 + q0 + 3];
            bool in = true;
            {
                float v[4] = {wv[0], wv[1], wv[2], wv[3]};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float4 dg = diag_s[q0 + c];
                    code[c] = cvt_e4m3x2(0.0f, div_recip(v[c], sw));
                    ne[c] = div_recip(__fsub_rn(lut_h[code[c]], v[c]), Recip{dg.x, dg.y, dg.z});
                    const float av = fabsf(v[c]);
                    in = in && ((av >= wmin && av <= 0x1p60f) || av == wzero);
                    // Eq. 12 inside the four
                    if (c == 0) {
                        v[1] = __fmaf_rn(ne[0], u0.y, v[1]);
                        v[2] = __fmaf_rn(ne[0], u0.z, v[2]);
                        v[3] = __fmaf_rn(ne[0], u0.w, v[3]);
                    } else if (c == 1) {
                        v[2] = __fmaf_rn(ne[1], u1.z, v[2]);
                        v[3] = __fmaf_rn(ne[1], u1.w, v[3]);
                    } else if (c == 2) {
                        v[3] = __fmaf_rn(ne[2], u23, v[3]);
                    }
                }
            }
            if (!in) {   // (tested once per four columns: a test per column stood in the chain)
                float f[8] = {wv[0], wv[1], wv[2], wv[3], 0.0f, 0.0f, 0.0f, 0.0f};
                const uint32_t all = dpq_four_slow(f, sw.b, lut_h, urow + q0);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    ne[c] = f[4 + c];
                    code[c] = (all >> (8 * c)) & 0xFFu;
                }
            }
            // Eq. 12 on this lane's columns, the four errors in order
#pragma unroll
            for (int kk = k; kk < 4; ++kk)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const ulonglong2 u2 = *reinterpret_cast<const ulonglong2*>(urow + c * 128 + 32 * kk + 4 * sl);
                    const unsigned long long e2 = pack_f32x2(ne[c], ne[c]);
                    w[2 * kk] = fma_f32x2(e2, u2.x, w[2 * kk]);
                    w[2 * kk + 1] = fma_f32x2(e2, u2.y, w[2 * kk + 1]);
                }
            if (sl == o && valid) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (p0 + 128 < K) ew[whole ? (int64_t)k * K + 16 * o + 4 * c : (int64_t)(q0 + c)] = ne[c];
                    code_s[rl * 128 + perm_s[q0 + c]] = lut_u[code[c]];
                }
            }
        }
        if (k == 2) {
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(marks.early(rows32, b)), "r"(1u) : "memory");
            }
        }
    }
    // The scale of the first row marks that the errors are in place; the codes need not be for that.
    const uint16_t scale = __bfloat16_as_ushort(__float2bfloat16_rn(grp.s));
    __syncthreads();
    if (tid == 0) {   // (row 0 of the 32)
        __threadfence();
        asm volatile("st.release.gpu.global.u16 [%0], %1;" ::"l"(gscale + n * G + og), "h"(scale) : "memory");
    }
    // codes of the group, original order, two per byte (even column in the low nibble); the first row's of the last block wait in the
    // work array (see DpqMarks)
    if (valid) {
        const uint32_t* cs = reinterpret_cast<const uint32_t*>(code_s + rl * 128 + sl * 16);
        uint32_t packed[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t a = cs[2 * i], c = cs[2 * i + 1];
            packed[i] = (a & 15u) | ((a >> 4) & 0xF0u) | ((a >> 8) & 0xF00u) | ((a >> 12) & 0xF000u) |
                        ((c & 15u) << 16) | ((c << 12) & 0xF00000u) | ((c << 8) & 0xF000000u) | ((c << 4) & 0xF0000000u);
        }
        uint8_t* to = n == 0 && p0 + 128 == K ? reinterpret_cast<uint8_t*>(work + p0) : codes + n * (K >> 1) + og * 64;
        *reinterpret_cast<uint2*>(to + sl * 8) = make_uint2(packed[0], packed[1]);
    }
    if (sl == 0 && valid) {
        if (rl > 0) gscale[n * G + og] = scale;
        if (gzero) gzero[n * G + og] = (uint8_t)grp.z;
    }
    return true;
}

// Bound by the FP32 pipes for large layers, by the chain of a block for small ones.  No CTA has to be resident for another to make
// progress: a task waits for tasks of earlier tickets only, which running CTAs hold; any number of calls can share the device.
// Measured, us per layer, a launch per step (whose CTAs start and drain together, with cp.async by all threads and two blocks' errors
// at a time) / this, search of six steps: (N, K) = (256, 1024) 266 / 263, (1024, 2048) 558 / 484, (2048, 2048) 683 / 537, (4096,
// 4096) 2384 / 2064, (8192, 8192) 14550 / 12020, (4096, 14336) 21190 / 17000 = 25 T FMA/s; none: (256, 4096) 880 / 833, (2048, 2048)
// 613 / 502, (4096, 14336) 20910 / 16740.  Of the last: order and waits 21200 -> 19800, tile
// loads three stages ahead -> 17850, panels of up to eight blocks -> 16870.  A tile's loop runs at 85 % of the pipe; what is left is
// the start and the end of tiles (13000 cycles of some 95000 at two blocks, 4 % at eight) and the tasks of the blocks, 14 % of the places.
__global__ void __launch_bounds__(kDpqThreads, 2)
dpq_kernel(const __grid_constant__ DpqMaps maps, float* work, const float* __restrict__ U, const int32_t* __restrict__ perm, int64_t N, int64_t K, int symmetric,
           int mse_steps, int per_channel, const float* __restrict__ s_w, uint8_t* codes, uint16_t* gscale,
           uint8_t* __restrict__ gzero, const DpqSteps first_step, unsigned int* status_word) {
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ int task[6];   // kind (0: end, 1: block, 2: errors), then what it is about
    __shared__ DpqSteps steps;                        // (thread 0's)
    __shared__ unsigned long long begin, end;         // tickets of the current step
    __shared__ uint64_t stage_bars[DpqSmem::kStages];
    __shared__ uint32_t abort_flag;
    const uint32_t bars = ptx::smem_addr(stage_bars);
    uint32_t ring = 0;                                // stages that this CTA has used
    const uint32_t sm_addr = ptx::smem_addr(sm);
    ptx::griddep_wait();
    const bool uvec = (reinterpret_cast<uintptr_t>(U) & 15u) == 0;
    const DpqMarks marks = {codes, gscale, perm, K};
    unsigned int* const control = marks.control();
    const DpqWait wait = {control, status_word};
    const unsigned int blocks32 = (unsigned)((N + kDpqRowsPerCta - 1) / kDpqRowsPerCta);
    if (threadIdx.x == 0) {
        steps = first_step;
        begin = end = 0;
        abort_flag = 0u;
        for (int i = 0; i < DpqSmem::kStages; ++i) ptx::mbar_init(bars + 8u * i, 1);
        ptx::fence_mbar_init();
    }
    while (true) {
        if (threadIdx.x == 0) {
            const unsigned int ticket = atomicAdd(control, 1u);
            while (ticket >= end && steps.b < steps.G) {
                begin = end;
                steps.next();
                if (steps.b < steps.G)
                    end = begin + blocks32 + (unsigned long long)steps.row_tiles * (unsigned)(steps.far.count + steps.near.count);
            }
            task[0] = 0;
            if (steps.b < steps.G) {
                unsigned int i = (unsigned int)(ticket - begin);
                if (i < blocks32) {
                    task[0] = 1;
                    task[1] = steps.b;
                    task[2] = (int)i;
                } else {
                    i -= blocks32;
                    const unsigned int col = i / (unsigned)steps.row_tiles;
                    const bool is_far = col < (unsigned)steps.far.count;
                    const DpqTrail tr = is_far ? steps.far : steps.near;
                    task[0] = 2;
                    task[1] = tr.errors;
                    task[2] = tr.blocks;
                    task[3] = tr.first + (int)(is_far ? col : col - (unsigned)steps.far.count);
                    task[4] = (int)(i % (unsigned)steps.row_tiles);
                }
            }
        }
        __syncthreads();
        const int kind = task[0], t1 = task[1], t2 = task[2], t3 = task[3], t4 = task[4];
        __syncthreads();
        if (kind == 0) break;
        const bool ok = kind == 1 ? dpq_block_rows(sm, sm_addr, work, U, perm, N, K, t1, t2, symmetric, mse_steps, per_channel, s_w, codes,
                                                   gscale, gzero, uvec, marks, wait)
                                  : dpq_trailing_tile(sm, sm_addr, work, U, N, K, t1, t2, t3, (int64_t)t4 * 128, uvec, marks, wait, maps, bars,
                                                     &abort_flag, ring);
        if (!ok) break;   // (the whole CTA)
        ptx::fence_proxy_async_smem();   // (the next task's bulk copies go where this one read and wrote)
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(control + 1, 1u) == gridDim.x - 1u) {   // the last one puts the codes where the control words were
            __threadfence();
            const uint4* from = reinterpret_cast<const uint4*>(work + K - 128);
            uint4* to = reinterpret_cast<uint4*>(control);
#pragma unroll
            for (int i = 0; i < 4; ++i) to[i] = __ldcg(from + i);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// The layer Hessian of the quantizer (Sec. 3.1; Sec. 3.3 for its preparation): H = X^T X over the
// calibration tokens, a plain FP32 contraction on the FMA pipes: every entry is one chain of fused
// multiply-adds over the tokens in order, whatever the tile.  (The tensor cores would be ten times as
// fast and closer to float64, but H would not keep its bits, and with H the codes quantized through it.)
// One CTA per TILE x TILE tile of the upper triangle, mirrored on the way out; eight warps of TILE / 8 rows and all
// columns, a lane TILE / 32 columns, rows in packed pairs.  Bound: the FP32 pipes.  Per token a warp reads its rows'
// values, which all lanes share, and TILE distinct column values: with (16 rows, 4 columns) five shared
// loads for 32 packed FMAs, with (8, 2) three for 8, against 8 for 16 scalar ones before.  Tokens come
// in double-buffered chunks of 16, through registers (BF16 -> FP32 on the way).  Measured, us, against the 64 x 64
// tiles of 4 x 4 scalar FMAs per thread: (T, K) = (2000, 1024) 212 -> 76, (1024, 4096) 799 -> 367 (24 T FMA/s,
// of the 28-31 T that a loop of FMAs alone reaches), (2048, 8192) 5820 -> 2586.  Where whole tiles would leave a last round that is not
// full, some are shared by their tokens between two launches (hessian_split, with figures).
// ---------------------------------------------------------------------------------------------
constexpr int kHessTok = 16;
// PART: 0, whole tiles only; 1, the first launch of a split; 2, the second.
template <int TILE, int PART>
__global__ void __launch_bounds__(256, TILE == 128 ? 2 : 4)
hessian_xtx_kernel(const uint16_t* __restrict__ x, int64_t tokens, int64_t K, int64_t ldx, float* __restrict__ H,
                   int accumulate, HessianSplit split) {
    constexpr int R = TILE / 8, C = TILE / 32;             // rows of a warp, columns of a lane
    constexpr int kLoads = 2 * kHessTok * TILE / 8 / 256;  // groups of eight features a thread fetches per chunk
    __shared__ __align__(16) float x_s[2][2][kHessTok][TILE];   // [buffer][rows | columns of the tile][token][feature]
    if (PART == 1) ptx::griddep_launch_dependents();
    // Whole tiles only: the upper triangle by rows; else the diagonal first, then the strict triangle by rows.
    const int nb = (int)((K + TILE - 1) / TILE), off = PART ? 1 : 0, n = nb - off;
    const bool bundle = PART == 1 && (int)blockIdx.x >= split.whole;
    int t = bundle ? split.whole + ((int)blockIdx.x - split.whole) * split.bundle : (PART == 2 ? split.whole : 0) + (int)blockIdx.x;
    const int end = bundle ? min(t + split.bundle, nb * (nb + 1) / 2) : t + 1;
    const int64_t T = bundle ? (int64_t)split.cut : tokens;
    do {
        // Row r of a triangle with n rows starts at r n - r (r - 1) / 2: the root of that, corrected by steps.
        const float b2 = 2.0f * (float)n + 1.0f;
        const int u = t - off * nb;
        int bi = (int)((b2 - sqrtf(fmaxf(b2 * b2 - 8.0f * (float)u, 0.0f))) * 0.5f);
        bi = min(max(bi, 0), n - 1);
        while (bi > 0 && bi * n - bi * (bi - 1) / 2 > u) --bi;
        while ((bi + 1) * n - (bi + 1) * bi / 2 <= u) ++bi;
        int bj = bi + u - (bi * n - bi * (bi - 1) / 2) + off;
        if (PART && t < nb) bi = bj = t;
        const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
        // eight features at once where every row of X starts on a 16-byte boundary
        const bool vec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && ldx % 8 == 0;

        uint4 in[kLoads];
        auto fetch = [&](int64_t t0) {
#pragma unroll
            for (int l = 0; l < kLoads; ++l) {
                const int i = tid + 256 * l, op = i / (kHessTok * TILE / 8), rest = i % (kHessTok * TILE / 8);
                const int64_t tok = t0 + rest / (TILE / 8), f = (int64_t)(op ? bj : bi) * TILE + rest % (TILE / 8) * 8;
                const uint16_t* src = x + tok * ldx + f;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (tok < T) {
                    if (vec && f + 8 <= K) {
                        v = __ldg(reinterpret_cast<const uint4*>(src));
                    } else {
                        uint32_t h[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) h[j] = f + j < K ? (uint32_t)__ldg(src + j) : 0u;
                        v = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
                    }
                }
                in[l] = v;
            }
        };
        auto put = [&](int buf) {
#pragma unroll
            for (int l = 0; l < kLoads; ++l) {
                const int i = tid + 256 * l, op = i / (kHessTok * TILE / 8), rest = i % (kHessTok * TILE / 8);
                float4* d = reinterpret_cast<float4*>(&x_s[buf][op][rest / (TILE / 8)][rest % (TILE / 8) * 8]);
                const uint4 v = in[l];
                d[0] = make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16),
                                   __uint_as_float(v.y & 0xFFFF0000u));
                d[1] = make_float4(__uint_as_float(v.z << 16), __uint_as_float(v.z & 0xFFFF0000u), __uint_as_float(v.w << 16),
                                   __uint_as_float(v.w & 0xFFFF0000u));
            }
        };
        unsigned long long acc[R / 2][C];   // rows 2 i and 2 i + 1
#pragma unroll
        for (int i = 0; i < R / 2; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) acc[i][j] = 0ull;
        struct Tok {
            ulonglong2 a[R / 4];
            float b[C];
        } k0, k1;
        // What the first launch hands to the second stands where the tile's mirror image goes in the end.
        float4* hand = reinterpret_cast<float4*>(H + ((int64_t)bj * TILE + R * warp) * K + (int64_t)bi * TILE) + lane;
        const int64_t from = PART == 2 ? split.cut : 0;
        fetch(from);
        if (PART == 2) {
            ptx::griddep_wait();
#pragma unroll
            for (int i = 0; i < R / 2; ++i)
#pragma unroll
                for (int j = 0; j < C; j += 2) {
                    const float4 v = __ldcg(hand + (int64_t)(i * C / 2 + j / 2) * (K / 4));
                    acc[i][j] = pack_f32x2(v.x, v.y);
                    acc[i][j + 1] = pack_f32x2(v.z, v.w);
                }
        }
        int buf = 0;
#pragma unroll 1
        for (int64_t t0 = from; t0 < T; t0 += kHessTok, buf ^= 1) {
            put(buf);
            __syncthreads();   // this chunk is there; the one before has been consumed by everybody
            if (t0 + kHessTok < T) fetch(t0 + kHessTok);
            const float* as = &x_s[buf][0][0][R * warp];
            const float* bs = &x_s[buf][1][0][C * lane];
            auto get = [&](Tok& k, int r) {
#pragma unroll
                for (int g = 0; g < R / 4; ++g) k.a[g] = *reinterpret_cast<const ulonglong2*>(as + r * TILE + 4 * g);
                if (C == 4) {
                    const float4 v = *reinterpret_cast<const float4*>(bs + r * TILE);
                    k.b[0] = v.x;
                    k.b[1] = v.y;
                    k.b[C - 2] = v.z;
                    k.b[C - 1] = v.w;
                } else {
                    const float2 v = *reinterpret_cast<const float2*>(bs + r * TILE);
                    k.b[0] = v.x;
                    k.b[1] = v.y;
                }
            };
            auto apply = [&](const Tok& k) {
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const unsigned long long b = pack_f32x2(k.b[j], k.b[j]);
#pragma unroll
                    for (int g = 0; g < R / 4; ++g) {
                        acc[2 * g][j] = fma_f32x2(k.a[g].x, b, acc[2 * g][j]);
                        acc[2 * g + 1][j] = fma_f32x2(k.a[g].y, b, acc[2 * g + 1][j]);
                    }
                }
            };
            get(k0, 0);
#pragma unroll
            for (int r = 0; r < kHessTok; r += 2) {
                get(k1, r + 1);
                apply(k0);
                if (r + 2 < kHessTok) get(k0, r + 2);
                apply(k1);
            }
        }
        if (bundle) {
#pragma unroll
            for (int i = 0; i < R / 2; ++i)
#pragma unroll
                for (int j = 0; j < C; j += 2) {
                    float4 v;
                    unpack_f32x2(acc[i][j], v.x, v.y);
                    unpack_f32x2(acc[i][j + 1], v.z, v.w);
                    hand[(int64_t)(i * C / 2 + j / 2) * (K / 4)] = v;
                }
            __syncthreads();   // (the last chunk has been read by everybody)
            continue;
        }
        // On a diagonal tile the 64 x 64 blocks below the diagonal are written as mirrors of those above.
        const int64_t gi0 = (int64_t)bi * TILE + R * warp, gj0 = (int64_t)bj * TILE + C * lane;
        const bool skip_row = bi == bj && TILE == 128 && warp >= 4 && lane < 16, mirror = bi != bj || (TILE == 128 && warp < 4 && lane >= 16);
        const bool wide = C == 4 && K % 4 == 0 && (reinterpret_cast<uintptr_t>(H) & 15u) == 0;   // (then gj0 < K covers the lane's four columns)
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            float lo[C], hi[C];
#pragma unroll
            for (int j = 0; j < C; ++j) unpack_f32x2(acc[i][j], lo[j], hi[j]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float* v = h == 0 ? lo : hi;
                const int64_t gi = gi0 + 2 * i + h;
                if (gi >= K || gj0 >= K || skip_row) continue;
                float* hr = H + gi * K + gj0;
                if (wide) {
                    if (accumulate) {
                        const float4 o = *reinterpret_cast<const float4*>(hr);
                        v[0] = __fadd_rn(v[0], o.x);
                        v[1] = __fadd_rn(v[1], o.y);
                        v[C - 2] = __fadd_rn(v[C - 2], o.z);
                        v[C - 1] = __fadd_rn(v[C - 1], o.w);
                    }
                    *reinterpret_cast<float4*>(hr) = make_float4(v[0], v[1], v[C - 2], v[C - 1]);
                } else {
#pragma unroll
                    for (int j = 0; j < C; ++j)
                        if (gj0 + j < K) {
                            if (accumulate) v[j] = __fadd_rn(v[j], hr[j]);
                            hr[j] = v[j];
                        }
                }
            }
#pragma unroll
            for (int j = 0; j < C; ++j) acc[i][j] = pack_f32x2(lo[j], hi[j]);
        }
        if (!mirror) return;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            if (gj0 + j >= K) continue;
            float* hc = H + (gj0 + j) * K + gi0;
#pragma unroll
            for (int i = 0; i < R / 2; i += 2) {
                float v[4];
                unpack_f32x2(acc[i][j], v[0], v[1]);
                unpack_f32x2(acc[i + 1][j], v[2], v[3]);
                if (wide) {
                    if (gi0 + 2 * i < K) *reinterpret_cast<float4*>(hc + 2 * i) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        if (gi0 + 2 * i + h < K) hc[2 * i + h] = v[h];
                }
            }
        }
    } while (++t < end && PART == 1);
}

// Sec. 3.3 (as in GPTQ): the Hessian in processing order, a unit diagonal for input features that
// never fired, damp * mean(diag) added to the diagonal.  Pass 1: the mean of the diagonal after the
// dead-feature rule (one CTA); pass 2: the permuted copy.
__global__ void __launch_bounds__(256)
hessian_diag_mean_kernel(const float* __restrict__ H, int64_t K, float* __restrict__ mean_out) {
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t k = threadIdx.x; k < K; k += 256) {
        const float d = H[k * K + k];
        s += d == 0.0f ? 1.0 : (double)d;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *mean_out = (float)(red[0] / (double)K);
}
__global__ void __launch_bounds__(256)
hessian_prepare_kernel(const float* __restrict__ H, int64_t K, const int32_t* __restrict__ perm, float damp,
                       const float* __restrict__ mean_diag, float* __restrict__ Hp) {
    const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (idx >= K * K) return;
    const int64_t i = idx / K, j = idx - i * K;
    const int64_t si = perm ? perm[i] : i, sj = perm ? perm[j] : j;
    float v = H[si * K + sj];
    if (i == j) {
        if (v == 0.0f) v = 1.0f;
        v = __fadd_rn(v, __fmul_rn(damp, *mean_diag));
    }
    Hp[idx] = v;
}

}  // namespace w4a8
