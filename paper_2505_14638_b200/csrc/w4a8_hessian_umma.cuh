// The layer Hessian of the quantizer (Sec. 3.1), H = X^T X over BF16 calibration tokens, on the tensor
// cores: tcgen05 kind::f16 MMAs with both operands read feature-major (the reduction runs over the
// tokens, whose rows are the slow dimension of X).
//
// Precision.  A product of two BF16 values is exact in FP32.  The tensor core adds them in FP32 but
// truncates, so a long chain inside the accumulator drifts below the true sum (T = 4096: 1.3e-5); only
// the TOK tokens of one stage (two or four MMAs) are therefore summed there, and the stages are added
// up in registers with round-to-nearest FP32 adds.  Relative error (2-norm) against float64, this kernel /
// the FP32 FMA chain of hessian_xtx_kernel: T = 63 4.7e-8 / 7.0e-8, 129 7.2e-8 / 8.9e-8,
// 256 1.0e-7 / 5.0e-7, 1024 1.0e-7 / 2.2e-6, 4096 1.6e-7 / 5.5e-6.
//
// What bounds it: the SM's L2 port.  A tile of 128 x 128 features pulls 32 KB per 64 tokens, 512
// cycles of that port (64 B per clock) against 256 of the tensor pipe, and moves 64 KB (128 KB with
// the mirrored half) of H on its way out.  Two CTAs per SM (one tile each, 96 KB of ring) let the
// epilogue of one tile run beside the loads of the other.  (T, K) = (1024, 4096): 34 us, 43 us when added
// to an earlier H, against 796 us on the FP32 FMA pipes; (4096, 8192): 372 us against 11.8 ms.
#pragma once

#include <cuda_bf16.h>

#include "w4a8_ptx.cuh"

namespace w4a8 {

template <int TOK_>
struct HessCfg {
    static constexpr int TILE = 128;               // features per tile, both ways
    static constexpr int TOK = TOK_;               // tokens per stage
    static constexpr int STAGES = 192 / TOK_;
    static constexpr int kPanel = TOK * 128;       // 64 features x TOK tokens: TOK rows of 128 bytes, 128-byte swizzle
    static constexpr int kOperand = 2 * kPanel;
    static constexpr int kStage = 2 * kOperand;
    static constexpr int kOutPitch = TILE + 1;     // floats; odd, so that columns and rows of the staged tile are conflict-free
    static constexpr int kRing = STAGES * kStage;
    static constexpr int kBarBytes = 256;
    static constexpr int kSmemBytes = kRing + kBarBytes + 1024;
    static constexpr int kEpiWarps = 8;
    static constexpr int kThreads = 64 + 32 * kEpiWarps;
    static_assert(TILE * kOutPitch * 4 <= kRing, "the finished tile is staged in the idle ring");
    static_assert((2 * STAGES + 5) * 8 + 8 <= kBarBytes, "barrier area");
};

namespace hess {
// Shared-memory matrix descriptor of an MN-major operand with the 128-byte swizzle: 64 features are one
// row of 128 bytes, eight tokens (rows) are one 1024-byte pattern; the next eight tokens are 1024
// bytes further, the next 64 features one panel further.
__device__ __forceinline__ uint64_t desc_mn_sw128(uint32_t addr, int panel) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((uint32_t)panel >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
}  // namespace hess

// Tile (bi, bj), bj >= bi, of the upper triangle per CTA.  CTA = ten warps: TMA producer, MMA issuer,
// eight that add the chunks up (lane quarter warp & 3, 64 of the 128 columns each) and store.
template <int TOK>
__global__ void __launch_bounds__(HessCfg<TOK>::kThreads, 2)
hessian_umma_kernel(const __grid_constant__ CUtensorMap tmap_x,  // X as bytes u8 [T][2 K], box 128 x TOK, 128B swizzle
                    int64_t T, int64_t K, float* __restrict__ H, int accumulate, unsigned int* status_word) {
    using C = HessCfg<TOK>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = ptx::smem_addr(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - raw_addr);
    const uint32_t bars = base + C::kRing;
    auto bar_full = [&](int s) { return bars + 8u * (uint32_t)s; };
    auto bar_empty = [&](int s) { return bars + 8u * (uint32_t)(C::STAGES + s); };
    auto bar_acc_full = [&](int b) { return bars + 8u * (uint32_t)(2 * C::STAGES + b); };
    auto bar_acc_empty = [&](int b) { return bars + 8u * (uint32_t)(2 * C::STAGES + 2 + b); };
    const uint32_t bar_drain = bars + 8u * (uint32_t)(2 * C::STAGES + 4);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + C::kRing + (2 * C::STAGES + 5) * 8);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nb = (int)((K + C::TILE - 1) / C::TILE);
    // row bi of the upper triangle starts at tile bi nb - bi (bi - 1) / 2: the root of that, corrected by a step
    const int t = (int)blockIdx.x;
    const float b2 = 2.0f * (float)nb + 1.0f;
    int bi = (int)((b2 - sqrtf(fmaxf(b2 * b2 - 8.0f * (float)t, 0.0f))) * 0.5f);
    bi = min(max(bi, 0), nb - 1);
    while (bi > 0 && bi * nb - bi * (bi - 1) / 2 > t) --bi;
    while ((bi + 1) * nb - (bi + 1) * bi / 2 <= t) ++bi;
    const int bj = bi + t - (bi * nb - bi * (bi - 1) / 2);
    const bool diag = bi == bj;
    const int nst = (int)((T + C::TOK - 1) / C::TOK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            ptx::mbar_init(bar_full(s), 1);
            ptx::mbar_init(bar_empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(bar_acc_full(b), 1);
            ptx::mbar_init(bar_acc_empty(b), 32 * C::kEpiWarps);
        }
        ptx::mbar_init(bar_drain, 1);
        *abort_flag = 0u;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_x);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), 2 * C::TILE);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        bool ok = true;
        int issued = 0;
        ptx::Ring r;
        const uint32_t bytes = diag ? (uint32_t)C::kOperand : (uint32_t)C::kStage;
        for (int it = 0; it < nst; ++it) {
            if (it >= C::STAGES) ok = ptx::mbar_wait(bar_empty(r.idx), r.phase ^ 1u, abort_flag, status_word);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            const uint32_t dst = base + (uint32_t)(r.idx * C::kStage);
            const uint32_t bar = bar_full(r.idx);
            if (ptx::elect_one()) {
                ptx::mbar_arrive_expect_tx(bar, bytes);
                ptx::tma_load_2d(dst, &tmap_x, bi * 256, it * C::TOK, bar);
                ptx::tma_load_2d(dst + C::kPanel, &tmap_x, bi * 256 + 128, it * C::TOK, bar);
                if (!diag) {
                    ptx::tma_load_2d(dst + C::kOperand, &tmap_x, bj * 256, it * C::TOK, bar);
                    ptx::tma_load_2d(dst + C::kOperand + C::kPanel, &tmap_x, bj * 256 + 128, it * C::TOK, bar);
                }
            }
            __syncwarp();
            issued = it + 1;
            r.advance(C::STAGES);
        }
        if (!ok) {
            // Gave up: let the copies already in flight land before the CTA goes away.
            for (int it = (issued > C::STAGES ? issued - C::STAGES : 0); it < issued; ++it) {
                const uint64_t t0 = ptx::globaltimer_ns();
                while (!ptx::mbar_try_wait(bar_full(it % C::STAGES), (uint32_t)((it / C::STAGES) & 1)) &&
                       ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // both operands BF16 and MN-major (bits 15, 16)
        constexpr uint32_t idesc = ptx::umma_idesc_bf16_f32(C::TILE, C::TILE) | (1u << 15) | (1u << 16);
        bool ok = true;
        ptx::Ring r;
        for (int c = 0; c < nst; ++c) {
            const int b = c & 1;
            if (c >= 2) ok = ptx::mbar_wait(bar_acc_empty(b), (uint32_t)(((c >> 1) - 1) & 1), abort_flag, status_word);
            ok = ok && ptx::mbar_wait(bar_full(r.idx), r.phase, abort_flag, status_word);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            const uint32_t a0 = base + (uint32_t)(r.idx * C::kStage);
            const uint64_t da = hess::desc_mn_sw128(a0, C::kPanel);
            const uint64_t db = hess::desc_mn_sw128(a0 + (diag ? 0u : (uint32_t)C::kOperand), C::kPanel);
            if (ptx::elect_one()) {
#pragma unroll
                for (int k = 0; k < C::TOK / 16; ++k)   // sixteen tokens = 2048 bytes further
                    ptx::umma_bf16(tmem_base + (uint32_t)(b * C::TILE), da + (uint64_t)(k * 128), db + (uint64_t)(k * 128),
                                   idesc, k > 0 ? 1u : 0u);
                ptx::umma_commit(bar_empty(r.idx));
                ptx::umma_commit(bar_acc_full(b));
            }
            __syncwarp();
            r.advance(C::STAGES);
        }
        if (!ok) {
            // Gave up: wait (bounded) for the MMAs already issued before tensor memory is freed.
            if (ptx::elect_one()) ptx::umma_commit(bar_drain);
            __syncwarp();
            const uint64_t t0 = ptx::globaltimer_ns();
            while (!ptx::mbar_try_wait(bar_drain, 0u) && ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs) {
            }
        }
    } else {
        // ------------------------------------------------------------------ chunk sums, then the tile on its way out
        const int q = warp & 3, ew = warp - 2, half = ew >> 2;
        const uint32_t lanes = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 64);
        float acc[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) acc[j] = 0.0f;
        const int64_t gi0 = (int64_t)bi * C::TILE, gj0 = (int64_t)bj * C::TILE;
        if (accumulate) {
            // the old values are wanted at the end: towards L2 now (two threads per row of the tile)
            const int64_t gi = gi0 + ((int)threadIdx.x - 64) / 2, gj = gj0 + ((int)threadIdx.x & 1) * 64;
            if (gi < K && gj < K) {
                ptx::prefetch_l2(H + gi * K + gj);
                if (gj + 32 < K) ptx::prefetch_l2(H + gi * K + gj + 32);
            }
        }
        bool ok = true;
        for (int c = 0; c < nst; ++c) {
            const int b = c & 1;
            ok = ptx::mbar_wait(bar_acc_full(b), (uint32_t)((c >> 1) & 1), abort_flag, status_word);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            ptx::tc_fence_after_sync();
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                uint32_t v[16];
                ptx::tmem_ld_32x32b_x16(lanes + (uint32_t)(b * C::TILE + g * 16), v);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[g * 16 + j] = __fadd_rn(acc[g * 16 + j], __uint_as_float(v[j]));
            }
            ptx::tc_fence_before_sync();
            ptx::mbar_arrive(bar_acc_empty(b));
        }
        // (the last chunk is complete: every stage has been consumed, the ring is idle)
        float* out = reinterpret_cast<float*>(sm);   // out[column][row], pitch kOutPitch
        if (ok) {
            const int row = q * 32 + lane;
#pragma unroll
            for (int j = 0; j < 64; ++j) out[(half * 64 + j) * C::kOutPitch + row] = acc[j];
        }
        // (all epilogue threads, also after giving up: the barrier counts them)
        asm volatile("bar.sync 1, %0;" ::"r"(32 * C::kEpiWarps) : "memory");
        ok = ok && *abort_flag == 0u;
        if (ok) {
            // rows of the tile, a warp per row: H[i][j], old value added.  On a diagonal tile the 64 x 64 block
            // below the diagonal is written as the mirror of the one above (a Hessian has no other).
            // Eight rows at a time: 32 loads in flight (one row at a time, the sixteen round trips of a warp
            // took as long as the main loop: 62 against 43 us at T = 1024, K = 4096).
#pragma unroll 1
            for (int i0 = ew; i0 < C::TILE; i0 += 8 * C::kEpiWarps) {
                float old[8][4];
                if (accumulate) {
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) {
                            const int64_t gi = gi0 + i0 + r * C::kEpiWarps, gj = gj0 + jj * 32 + lane;
                            old[r][jj] = (gi < K && gj < K) ? H[gi * K + gj] : 0.0f;
                        }
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int i = i0 + r * C::kEpiWarps;
                    const int64_t gi = gi0 + i;
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        const int j = jj * 32 + lane;
                        if (gi >= K || gj0 + j >= K || (diag && (i >> 6) > (jj >> 1))) continue;
                        float v = out[j * C::kOutPitch + i];
                        if (accumulate) {
                            v = __fadd_rn(v, old[r][jj]);
                            out[j * C::kOutPitch + i] = v;
                        }
                        H[gi * K + gj0 + j] = v;
                    }
                }
            }
        }
        asm volatile("bar.sync 1, %0;" ::"r"(32 * C::kEpiWarps) : "memory");
        if (ok) {
            // the mirrored tile, a warp per row: H[j][i]
            for (int j = (diag ? 64 : 0) + ew; j < C::TILE; j += C::kEpiWarps) {
                const int64_t gj = gj0 + j;
                if (gj >= K) break;
                float* hrow = H + gj * K + gi0;
#pragma unroll
                for (int ii = 0; ii < 4; ++ii) {
                    const int i = ii * 32 + lane;
                    if (gi0 + i >= K || (diag && i >= 64)) continue;
                    hrow[i] = out[j * C::kOutPitch + i];
                }
            }
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, 2 * C::TILE);
    }
}

}  // namespace w4a8
