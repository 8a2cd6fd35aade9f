// W4A8 linear for few tokens, one layer per launch: the packed weights go from global memory straight
// into the registers of the warps that multiply them.
//
// What bounds a small layer at a few tokens is not the HBM rate but everything around it: a launch of the
// kernels that stage weights through shared memory and tensor memory spends three to four
// microseconds on barriers, allocation, the first hand-overs between its roles and the drain, longer than the
// weights of a 4096 x 4096 layer take to arrive.  Here a warp fetches 16 rows x four k-blocks (4 KB of
// codes, eight 16-byte loads per lane), expands them in registers (Eq. 10, one table per row and k-block) and
// feeds them to mma.sync m16n8k32 E4M3 MMAs (FP32 accumulation): no copies, no barriers until the row tile is
// done.  (1024, 1024) at M = 8: 3.4 us against 6.3 (the linear layer alone).  For larger layers the integer pipe is taken to be
// the bound: this form of the MMA has its FP8 operands converted to 16 bits, two conversions for each of the six operand
// registers of an MMA, 192 per 16 rows x 512 columns and eight tokens, beside some 250 instructions of expansion (both counted
// from this source, not measured); the tcgen05 kernels are spared the former: (28672, 4096) at M = 8 22 us against 17.5.
//
// Fragment layout.  The order of the reduction index is free as long as both operands share it: the four
// lanes of a row take four different k-blocks (a lane owns all 128 weights of its row and k-block: one table
// per 128 weights), and word j of every lane's 16 words -- eight weights, the two K = 4 pieces that an
// A fragment holds per row -- is multiplied with the eight activation bytes of the same columns, which the lane of
// the B fragment with the same index finds side by side.  So neither operand is shuffled.
//
// A CTA (16 warps, one per SM) takes a contiguous run of 8-row units and the whole K; its activations sit
// in shared memory.
// Warps are arranged as Tc row tiles x Wq shares of the k-block quads; the Wq partial sums of a tile are
// added in shared memory in ascending order (results repeat bit for bit), scaled (Eq. 4, Eq. 11) and stored.
//
// Launched with programmatic stream serialization; prepacked weights, which depend on no earlier kernel,
// are requested before griddepcontrol.wait, everything else after it.
#pragma once

#include <cuda_bf16.h>

#include "w4a8_ptx.cuh"
#include "w4a8_tiled_format.cuh"

namespace w4a8 {

template <int FMT_, int NT_>
struct DirCfg {
    static constexpr int FMT = FMT_;
    static constexpr int NT = NT_;                 // token tiles of eight
    static constexpr int kWarps = 16;
    static constexpr int kThreads = 32 * kWarps;
    static constexpr int kPitch = 20;              // floats per token of a partial tile of 16 rows (spreads the fragments over the banks)
    static_assert(NT == 1 || NT == 2, "up to sixteen tokens");
};

namespace direct {
__device__ __forceinline__ void mma_e4m3(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.f32.e4m3.e4m3.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 ld_weights(const uint8_t* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w)); }
}  // namespace direct

template <class Cfg>
__global__ void __launch_bounds__(Cfg::kThreads, 1)
linear_direct_kernel(const uint8_t* __restrict__ x8, int64_t ldx8, const uint8_t* __restrict__ weights,
                     const uint16_t* __restrict__ gscale, const uint8_t* __restrict__ gzero,  // canonical format only
                     const float* __restrict__ s_x, const float* __restrict__ s_w, int sw_stride,
                     void* __restrict__ y, int64_t ldy, int out_dtype, int M, int N, int K, const DirPlan plan) {
    constexpr int FMT = Cfg::FMT, NT = Cfg::NT;
    constexpr bool kCanonical = FMT == kFmtCanonical, kSignMag = FMT == kFmtTiledSignMag;
    constexpr int MB = kCanonical ? 0 : meta_bytes(FMT);
    extern __shared__ __align__(16) uint8_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
    const int KB = K >> 7, Q = (KB + 3) >> 2;
    const int NU = N >> 3;
    const int u0 = (int)((int64_t)blockIdx.x * NU / plan.P), u1 = (int)((int64_t)(blockIdx.x + 1) * NU / plan.P);
    const int T = (u1 - u0 + 1) >> 1;   // row tiles: two units, the last one perhaps alone
    const int Wq = plan.Wq, Tc = plan.Tc;
    const int tc = warp / Wq, wq = warp - tc * Wq;
    const bool works = tc < Tc && tc < T;
    uint8_t* xs = sm;
    float* sx_s = reinterpret_cast<float*>(sm + (size_t)M * plan.xpitch);
    float* red = sx_s + ((M + 3) & ~3);

    ptx::griddep_launch_dependents();
    if constexpr (kCanonical) ptx::griddep_wait();

    // The unit of work (tile t, quad q): rows gid of either 8-row unit, k-block 4 q + tig.  Where a k-block or the second
    // 8-row unit does not exist, the last or first one is read in its place and its scale is taken as zero: zero weights.
    const uint8_t* meta0 = weights + (int64_t)KB * N * kRowCodeBytes;
    uint4 lo[4], hi[4];
    uint32_t mlo = kZeroMeta<FMT>, mhi = kZeroMeta<FMT>;   // scale (BF16 bits), zero-point above it
    struct Unit {
        const uint8_t* lo;
        const uint8_t* hi;
    };
    auto unit = [&](int t, int q) {
        const int kb = min(4 * q + tig, KB - 1), n = (u0 + 2 * t) * 8 + gid;
        const bool has_hi = u0 + 2 * t + 1 < u1;
        Unit u;
        if constexpr (kCanonical) {
            u.lo = weights + (int64_t)n * (K >> 1) + kb * 64;
            u.hi = u.lo + (has_hi ? (int64_t)8 * (K >> 1) : 0);
        } else {
            u.lo = weights + ((int64_t)kb * N + (n - gid)) * kRowCodeBytes + gid * 16;
            u.hi = u.lo + (has_hi ? 8 * kRowCodeBytes : 0);
        }
        return u;
    };
    auto load_chunk = [&](const Unit& u, int c) {
        if constexpr (kCanonical) {   // (the four 16-byte pieces of a row's 64 bytes meet in L1)
            lo[c] = __ldg(reinterpret_cast<const uint4*>(u.lo + c * 16));
            hi[c] = __ldg(reinterpret_cast<const uint4*>(u.hi + c * 16));
        } else {
            lo[c] = direct::ld_weights(u.lo + c * (int)kChunkStride);
            hi[c] = direct::ld_weights(u.hi + c * (int)kChunkStride);
        }
    };
    auto load_meta = [&](int t, int q, uint32_t& a, uint32_t& b) {
        const int kb = 4 * q + tig, n = (u0 + 2 * t) * 8 + gid;
        const bool in = kb < KB, in_hi = in && u0 + 2 * t + 1 < u1;
        a = b = kZeroMeta<FMT>;
        if constexpr (kCanonical) {
            const int64_t i = (int64_t)n * KB + kb, j = i + (int64_t)8 * KB;
            if (in) a = (uint32_t)__ldg(gscale + i) | (gzero ? (uint32_t)__ldg(gzero + i) : 8u) << 16;
            if (in_hi) b = (uint32_t)__ldg(gscale + j) | (gzero ? (uint32_t)__ldg(gzero + j) : 8u) << 16;
        } else {
            const uint8_t* p = meta0 + ((int64_t)kb * N + n) * MB;
            if constexpr (kSignMag) {
                if (in) a = (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(p));
                if (in_hi) b = (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(p + 8 * MB));
            } else {
                if (in) a = __ldg(reinterpret_cast<const uint32_t*>(p));
                if (in_hi) b = __ldg(reinterpret_cast<const uint32_t*>(p + 8 * MB));
            }
        }
    };
    int t = tc, q = wq;
    if (works) {
        load_meta(t, q, mlo, mhi);
        const Unit u = unit(t, q);
#pragma unroll
        for (int c = 0; c < 4; ++c) load_chunk(u, c);
    }
    if constexpr (!kCanonical) ptx::griddep_wait();
    {
        // activations: k-blocks 144 bytes apart, tokens an odd multiple of 64 bytes: the lanes (gid, tig) of a load phase
        // (two tokens, four k-blocks) then hit all banks, at constant offsets within a k-block
        const int pieces = K >> 4;
        const uint32_t xs_addr = ptx::smem_addr(xs);
        for (int i = threadIdx.x; i < M * pieces; i += Cfg::kThreads) {
            const int m = i / pieces, pc = i - m * pieces;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(xs_addr + (uint32_t)(m * plan.xpitch + (pc >> 3) * 144 + (pc & 7) * 16)),
                         "l"(x8 + (int64_t)m * ldx8 + pc * 16)
                         : "memory");
        }
        if ((int)threadIdx.x < M) sx_s[threadIdx.x] = __ldg(s_x + threadIdx.x);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
    if (!works) return;

    // this lane's activations: token min(8 j + gid, M - 1) (tokens past the end are computed and not stored)
    uint32_t xrow[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) xrow[j] = (uint32_t)(min(8 * j + gid, M - 1) * plan.xpitch);
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][i] = 0.0f;
    int buf = 0;
    while (true) {
        int tn = t, qn = q + Wq;   // the unit after this one
        const bool last_of_tile = qn >= Q;
        if (last_of_tile) {
            tn = t + Tc;
            qn = wq;
        }
        const bool more = tn < T;
        const uint32_t xoff = (uint32_t)(min(4 * q + tig, KB - 1) * 144);
        typename LutOf<FMT>::type llo, lhi;
        llo.build_meta(mlo);
        lhi.build_meta(mhi);
        if (more) load_meta(tn, qn, mlo, mhi);
        const bool has_hi = u0 + 2 * t + 1 < u1;
        const Unit next = unit(more ? tn : t, more ? qn : q);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t f[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};   // words 2 h, 2 h + 1 of the chunk: (low, high half) x (row gid, row gid + 8)
                llo.dequant8(direct::word(lo[c], 2 * h), f[0], f[2]);
                llo.dequant8(direct::word(lo[c], 2 * h + 1), f[4], f[6]);
                if (has_hi) {
                    lhi.dequant8(direct::word(hi[c], 2 * h), f[1], f[3]);
                    lhi.dequant8(direct::word(hi[c], 2 * h + 1), f[5], f[7]);
                }
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const uint4 x = *reinterpret_cast<const uint4*>(sm + (xrow[j] + xoff) + (2 * c + h) * 16);
                    direct::mma_e4m3(acc[j], f[0], f[1], f[2], f[3], x.x, x.y);
                    direct::mma_e4m3(acc[j], f[4], f[5], f[6], f[7], x.z, x.w);
                }
            }
            load_chunk(next, c);   // (after the last unit: read again, not used)
        }
        if (last_of_tile) {
            // partial tile of this warp: [token][row], then the Wq partial sums in ascending order
            const int n0 = (u0 + 2 * t) * 8;
            constexpr int kTile = 8 * NT * Cfg::kPitch;
            float* tile = red + (buf * Cfg::kWarps + tc * Wq) * kTile;
            float* mine = tile + wq * kTile;
            const int row_o = lane & 15;
            const bool row_ok = row_o < 8 || u0 + 2 * t + 1 < u1;
            const float swn = row_ok ? __ldg(s_w + (int64_t)(n0 + row_o) * sw_stride) : 0.0f;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                mine[(8 * j + 2 * tig) * Cfg::kPitch + gid] = acc[j][0];
                mine[(8 * j + 2 * tig + 1) * Cfg::kPitch + gid] = acc[j][1];
                mine[(8 * j + 2 * tig) * Cfg::kPitch + gid + 8] = acc[j][2];
                mine[(8 * j + 2 * tig + 1) * Cfg::kPitch + gid + 8] = acc[j][3];
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[j][i] = 0.0f;
            }
            if (Wq > 1)
                asm volatile("bar.sync %0, %1;" ::"r"(1 + tc), "r"(32 * Wq) : "memory");
            else
                __syncwarp();
            for (int m = 2 * wq + (lane >> 4); m < M; m += 2 * Wq) {
                float sum = 0.0f;
#pragma unroll 4
                for (int w = 0; w < Wq; ++w) sum += tile[w * kTile + m * Cfg::kPitch + row_o];
                const float res = sum * (sx_s[m] * swn);   // Eq. 4, Eq. 11
                if (row_ok) {
                    if (out_dtype == W4A8_OUT_FP32)
                        reinterpret_cast<float*>(y)[(int64_t)m * ldy + n0 + row_o] = res;
                    else
                        reinterpret_cast<__nv_bfloat16*>(y)[(int64_t)m * ldy + n0 + row_o] = __float2bfloat16_rn(res);
                }
            }
            buf ^= 1;   // two buffers: a warp gets to one again only behind the barrier of the tile in between
            if (Wq == 1) __syncwarp();
        }
        if (!more) break;
        t = tn;
        q = qn;
    }
}

}  // namespace w4a8
