// W4A8 linear layer for up to 128 tokens on prepacked layers of many output channels: every CTA takes one contiguous run of
// rows (an SM's share of the channels, up to 256 rows) and walks the whole K.
//
// Bound by the weight stream: a k-block of an SM's rows is some 13 KB, 0.29 us of HBM time, beside which its expansion (two warps
// of 32 rows per SM sub-partition, 200 cycles each), its MMAs (two row blocks of at most 4 x 64 cycles) and the activation tile
// (read once for both row blocks) all fit.  Cutting the channels into tiles of 128 instead leaves most SMs without a second
// tile: 224 tiles of a 28672-channel layer take 148 SMs two rounds.
//
// Data path of a k-block: bulk copies of codes and meta data into a ring in shared memory; one thread per row expands them
// (Eq. 10) into a slot of tensor memory (32 columns per block of 128 rows); MMAs with the weights as the A operand from there and
// the activation tile, N = tokens rounded up to sixteen, as B from shared memory; accumulators in tensor memory.  Two rings, as
// weights can be fetched and expanded far ahead while activations are still being quantized by the kernel before: packed
// weights (freed by the expansion), and expanded weights with their activation tile (freed by the MMAs).
//
// Warps: 0 activation tiles, 1 meta data (and tensor memory's allocation), 2 codes, 3 MMAs -- on the sub-partition whose lane
// quarter has the fewest rows; an MMA costs its sub-partition some 32 issue cycles --, then four groups of four that expand
// every fourth stage and drain the accumulators at the end.  A stage is two items of 128 rows x one k-block: both row blocks,
// or two k-blocks of the one there is.  (An issuing lane's round of waits and requests costs it 250-400 cycles beside warps
// that expand: stages of one item took (1, 14336, 4096) 11.7 us in place of 10.7.)  One CTA takes the SM's shared and tensor
// memory, and the registers left over let the quantization kernel between two layers run beside it, so that the next layer's
// CTAs fill their rings meanwhile (programmatic dependent launch).
//
// K cut (up to sixteen tokens, few channels): each CTA takes part of a run's k-blocks and leaves its sums in the workspace; the CTA
// that arrives last adds them in ascending order of the parts.  HALF: two expansion groups, half the shared and tensor
// memory, so that the CTAs of two launches share an SM and the second is set up and has expanded its first stages when its
// activations come, or the launch before is through: better only where a CTA walks a short K and the main loop does not hide
// that (half_rows_apply).
//
// Each accumulator is one chain of MMAs over K in ascending order: where K is not cut, the bits of a chain launch.
//
// Measured, quantization and linear layer back to back, weights not in L2, us, the kernels before (K walked by two groups on half
// an SM up to sixteen tokens; whole tiles above) / this: (8, 28672, 4096) 18.3 / 15.6, (16, 28672, 8192) 33.1 / 27.3 = 4.4 TB/s,
// (8, 4096, 14336) 14.8 / 13.3, (1, 14336, 4096) 11.1 / 9.9, (32, 28672, 4096) 21.8 / 16.0, (77, 28672, 4096) 23.5 / 18.0, (128, 28672,
// 8192) 50.5 / 37.7; with zero-points (8, 28672, 4096) 21.3 / 18.3, (64, 28672, 4096) 25.2 / 19.5.  Time stamps of (8, 28672, 4096):
// 3.8 us until the activations are there, 8.3 us of main loop at 510 cycles a k-block (its eight MMAs take 415 to issue, its
// expansion 420), 1.6 us of last MMAs, outputs and exit.
#pragma once

#include <cuda_bf16.h>

#include "w4a8_decode_plan.h"
#include "w4a8_ptx.cuh"
#include "w4a8_tiled_format.cuh"

namespace w4a8 {

template <int FMT_, bool HALF_ = false>
struct RowsCfg : RowsSizes<FMT_, HALF_> {
    static constexpr int FMT = FMT_;
    static constexpr bool HALF = HALF_;         // half an SM per CTA (see the kernel's comment)
    static constexpr int kThreads = 128 + 128 * RowsSizes<FMT_, HALF_>::G;
    // (registers: 80 a thread, 640 threads of them leave room for the quantization kernel's CTA beside them; so do 2 x 384)
    static constexpr int kBoundThreads = HALF_ ? kThreads : 768, kBoundCtas = HALF_ ? 2 : 1;
};

template <class Cfg>
__global__ void __launch_bounds__(Cfg::kBoundThreads, Cfg::kBoundCtas)
linear_rows_kernel(const __grid_constant__ CUtensorMap tmap_x,   // X8 u8 [M][K], box 128 x MN, 128B swizzle
                   const uint8_t* __restrict__ wpp, const float* __restrict__ s_x, const float* __restrict__ s_w, int sw_stride,
                   void* __restrict__ y, int64_t ldy, int out_dtype, int M, int N, int K, const RowsPlan plan,
                   unsigned int* counters, float* partials, unsigned int* status_word) {
    constexpr int G = Cfg::G, MB = Cfg::kMeta;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = ptx::smem_addr(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - raw_addr);

    const int S1 = plan.S1, S2 = plan.S2, RB = plan.RB, MN = plan.MN, T = plan.T;
    const int KS = 2 / RB;   // k-blocks per stage
    const uint32_t xtile = (uint32_t)MN * 128u, xslot = (uint32_t)KS * xtile, wslot = (uint32_t)(KS * plan.whalf);
    const uint32_t x_ring = base, w_ring = x_ring + (uint32_t)S2 * xslot;
    const uint32_t out_off = (uint32_t)S2 * xslot + (uint32_t)S1 * wslot;
    const uint32_t bars_off = out_off + (uint32_t)Cfg::kOutBytes, bars = base + bars_off;
    const uint32_t bar_wfull = bars, bar_wfree = bar_wfull + 8u * Cfg::kS1Max;             // packed weights landed / expanded
    const uint32_t bar_full = bar_wfree + 8u * Cfg::kS1Max, bar_free = bar_full + 8u * Cfg::kS2Max;   // stage ready for its MMAs / consumed
    const uint32_t bar_acc_full = bar_free + 8u * Cfg::kS2Max, bar_acc_empty = bar_acc_full + 8u, bar_drain = bar_acc_full + 16u;
    volatile uint32_t* tmem_slot =
        reinterpret_cast<volatile uint32_t*>(sm + bars_off + 8u * (2 * Cfg::kS1Max + 2 * Cfg::kS2Max + 3));
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* ticket = tmem_slot + 2;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Tile t: run t / cut of the rows, in units of eight, and part t % cut of the k-blocks.
    const int cut = plan.cut, part = (int)blockIdx.x % cut;   // (cut > 1: the grid has a CTA per tile)
    const int kb0 = part * (K >> 7) / cut, KB = (part + 1) * (K >> 7) / cut - kb0;
    const int NS = (KB + KS - 1) / KS;   // stages of a tile; the last one may hold one k-block
    auto first_unit = [&](int run) { return (int64_t)run * plan.units + min(run, plan.more); };
    const int p = blockIdx.x, P = gridDim.x;
    const int acols = (RB * MN + 31) & ~31;   // columns of the accumulators

    // Warp 2 sets up the barriers (one lane each), warp 1 allocates tensor memory.  Neither waits for the other or for the rest
    // of the CTA: they go on with their requests for weights, which need the barriers of the first ring only.
    if (warp == 2) {
        constexpr int kBars = 2 * Cfg::kS1Max + 2 * Cfg::kS2Max + 3, kF = 2 * Cfg::kS1Max, kE = kF + 2 * Cfg::kS2Max;
        for (int i = lane; i < kBars; i += 32) {
            uint32_t count = 1;                                  // a slot consumed, accumulators complete, drained after an abort
            if (i < Cfg::kS1Max) count = 2;                      // packed weights landed: codes, meta data
            else if (i < kF) count = 4;                          // expanded: the warps of a group
            else if (i < kF + Cfg::kS2Max) count = 4 + 1;        // ready for the MMAs: the same, and the activation tiles
            else if (i == kE + 1) count = 4 * G;                 // accumulators read
            ptx::mbar_init(bars + 8u * (uint32_t)i, count);
        }
        if (lane == 0) *abort_flag = 0u;
        ptx::fence_mbar_init();
        __syncwarp();
        asm volatile("bar.arrive 1, 64;" ::: "memory");   // warp 1 may use the barriers
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), Cfg::kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    if (warp == 1 || warp == 2) {
        asm volatile("bar.arrive 2, %0;" ::"n"(Cfg::kThreads) : "memory");
        if (warp == 1) asm volatile("bar.sync 1, 64;" ::: "memory");
    } else {
        if (threadIdx.x == 0) ptx::prefetch_tensormap(&tmap_x);
        asm volatile("bar.sync 2, %0;" ::"n"(Cfg::kThreads) : "memory");
    }
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = warp == 1 || warp == 2 ? 0u : *tmem_slot;   // (these two have not waited for it)
    ptx::griddep_launch_dependents();

    if (warp == 1 || warp == 2) {
        // ------------------------------------------------------------------ meta data / codes (whole warp, one lane issues)
        // (they depend on no earlier kernel)
        const uint32_t rowb = warp == 1 ? (uint32_t)MB : (uint32_t)kRowCodeBytes;
        const int64_t step = (int64_t)N * rowb;   // one k-block further
        const uint8_t* src0 = wpp + (warp == 1 ? (int64_t)(K >> 7) * N * kRowCodeBytes : 0) + kb0 * step;
        bool ok = true;
        ptx::Ring r;
        int issued = 0;
        for (int t = p; t < T && ok; t += P) {
            const int64_t u0 = first_unit(t / cut), u1 = first_unit(t / cut + 1);
            const uint32_t rows = (uint32_t)(u1 - u0) * 8u, bytes = rows * rowb;
            const uint32_t off = w_ring + (warp == 1 ? rows * kRowCodeBytes : 0u);
            const uint8_t* src = src0 + u0 * 8 * rowb;
            for (int st = 0; st < NS; ++st) {
                if (issued >= S1) ok = ptx::mbar_wait_warp(bar_wfree + 8u * r.idx, r.phase ^ 1u, abort_flag, status_word);
                if (!ok) break;
                const bool two = KS == 2 && 2 * st + 1 < KB;
                const uint32_t full = bar_wfull + 8u * r.idx, dst = off + (uint32_t)r.idx * wslot;
                if (ptx::elect_one()) {
                    ptx::mbar_arrive_expect_tx(full, two ? 2u * bytes : bytes);
                    ptx::bulk_load(dst, src, bytes, full);
                    if (two) ptx::bulk_load(dst + (uint32_t)plan.whalf, src + step, bytes, full);
                }
                src += KS * step;
                r.advance(S1);
                ++issued;
            }
        }
        if (!ok && lane == 0) {   // gave up: let the copies in flight land before the CTA goes away
            const uint64_t t0 = ptx::globaltimer_ns();
            for (int i = issued > S1 ? issued - S1 : 0; i < issued; ++i)
                while (!ptx::mbar_try_wait(bar_wfull + 8u * (i % S1), (uint32_t)((i / S1) & 1)) &&
                       ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs / 20) {
                }
        }
        __syncwarp();
    } else if (warp == 0) {
        // ------------------------------------------------------------------ activation tiles (whole warp, one lane issues)
        bool ok = true;
        ptx::Ring r;
        int issued = 0;
        ptx::griddep_wait();
        for (int t = p; t < T && ok; t += P)
            for (int st = 0; st < NS; ++st) {
                if (issued >= S2) ok = ptx::mbar_wait_warp(bar_free + 8u * r.idx, r.phase ^ 1u, abort_flag, status_word);
                if (!ok) break;
                const uint32_t full = bar_full + 8u * r.idx, dst = x_ring + (uint32_t)r.idx * xslot;
                const bool two = KS == 2 && 2 * st + 1 < KB;
                if (ptx::elect_one()) {
                    ptx::mbar_arrive_expect_tx(full, two ? xslot : xtile);
                    ptx::tma_load_2d(dst, &tmap_x, (kb0 + st * KS) * 128, 0, full);
                    if (two) ptx::tma_load_2d(dst + xtile, &tmap_x, (kb0 + st * KS + 1) * 128, 0, full);
                }
                r.advance(S2);
                ++issued;
            }
        if (!ok && lane == 0) {   // (the barriers count the expanding warps too, which may have given up as well)
            const uint64_t t0 = ptx::globaltimer_ns();
            for (int i = issued > S2 ? issued - S2 : 0; i < issued; ++i)
                while (!ptx::mbar_try_wait(bar_full + 8u * (i % S2), (uint32_t)((i / S2) & 1)) &&
                       ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs / 20) {
                }
        }
        __syncwarp();
    } else if (warp == 3) {
        // ------------------------------------------------------------------ MMAs (whole warp, one lane issues)
        bool ok = true;
        ptx::Ring r;
        uint32_t acc_phase = 0;
        const uint32_t idesc = ptx::umma_idesc_e4m3_f32(128, 0) | (uint32_t)(MN >> 3) << 17;
        const uint32_t b_lo0 = ptx::umma_desc_lo(x_ring), b_step = xslot >> 4, b_half = xtile >> 4;
        for (int t = p; t < T && ok; t += P) {
            if (t != p) {
                ok = ptx::mbar_wait_warp(bar_acc_empty, acc_phase, abort_flag, status_word);
                acc_phase ^= 1u;
            }
            for (int st = 0; st < NS && ok; ++st) {
                ok = ptx::mbar_wait_warp(bar_full + 8u * r.idx, r.phase, abort_flag, status_word);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t b_lo = b_lo0 + (uint32_t)r.idx * b_step, accumulate = st > 0 ? 1u : 0u;
                const uint32_t a_col = tmem_base + (uint32_t)(acols + r.idx * 64), done = bar_free + 8u * r.idx;
                const bool second = RB == 2 || (KS == 2 && 2 * st + 1 < KB);
                const uint32_t d1 = RB == 2 ? tmem_base + (uint32_t)MN : tmem_base, b_lo1 = RB == 2 ? b_lo : b_lo + b_half;
                if (ptx::elect_one()) {
                    ptx::umma_f8_kblock_ts(tmem_base, a_col, b_lo, idesc, accumulate);
                    if (second) ptx::umma_f8_kblock_ts(d1, a_col + 32u, b_lo1, idesc, RB == 2 ? accumulate : 1u);
                    ptx::umma_commit(done);
                }
                r.advance(S2);
            }
            if (ok && ptx::elect_one()) ptx::umma_commit(bar_acc_full);
        }
        if (!ok && lane == 0) {   // gave up: wait for the MMAs already issued before tensor memory is freed
            ptx::umma_commit(bar_drain);
            const uint64_t t0 = ptx::globaltimer_ns();
            while (!ptx::mbar_try_wait(bar_drain, 0u) && ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs) {
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ expansion, then the outputs
        const int g = (warp - 4) >> 2, q = warp & 3;   // (a warp reaches the tensor-memory lanes of its quarter)
        const uint32_t lanes = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t stage = base + out_off + (uint32_t)((warp - 4) * Cfg::kStageBytes);
        const int es = out_dtype == W4A8_OUT_FP32 ? 4 : 2;
        const bool wide = ((ldy * es) & 15) == 0;   // rows of Y 16-byte aligned (y itself is)
        const int chunks = (M + 15) >> 4;
        ptx::Ring r1, r2;   // this group's next stage in the two rings; every G-th is its own
        for (int i = 0; i < g; ++i) {
            r1.advance(S1);
            r2.advance(S2);
        }
        bool ok = true;
        uint32_t acc_phase = 0;
        int it = g;         // the same, counted over all runs
        int done_runs = 0;
        for (int t = p; t < T && ok; t += P) {
            const int64_t u0 = first_unit(t / cut);
            const int R = (int)(first_unit(t / cut + 1) - u0) * 8;
            const int row = q * 32;
            const bool has0 = row < R, has1 = RB == 2 ? 128 + row < R : has0;   // (warp-uniform) rows of the stage's two items
            // a lane past the last row repeats it: its tensor-memory lane feeds outputs that do not exist
            const int row0 = min(row + lane, R - 1), row1 = RB == 2 ? min(128 + row + lane, R - 1) : row0;
            const uint32_t next = RB == 2 ? 0u : (uint32_t)plan.whalf;          // (the second item: the next k-block)
            const uint32_t c0 = tiled_row_offset(row0), c1 = next + tiled_row_offset(row1);
            const uint32_t m0 = (uint32_t)(R * kRowCodeBytes + row0 * MB), m1 = next + (uint32_t)(R * kRowCodeBytes + row1 * MB);
            const int end = (done_runs + 1) * NS;
            for (; it < end; it += G) {
                // The stage's tensor-memory slot first: once its previous MMAs have completed, every earlier stage of
                // packed weights has landed, among them the previous one in this slot (S1 >= S2), so that "landed"
                // cannot be taken for the phase before; and S2 >= G keeps this group within one phase here.
                if (it >= S2) ok = ptx::mbar_wait_warp(bar_free + 8u * r2.idx, r2.phase ^ 1u, abort_flag, status_word);
                ok = ok && ptx::mbar_wait_warp(bar_wfull + 8u * r1.idx, r1.phase, abort_flag, status_word);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t w = w_ring + (uint32_t)r1.idx * wslot;
                const uint32_t a_col = lanes + (uint32_t)(acols + r2.idx * 64);
                if (has1 && (it + 1 < end || KB % KS == 0))
                    dequant_two_rows_to_tmem<Cfg::FMT>(w + c0, w + m0, w + c1, w + m1, a_col);
                else if (has0)
                    dequant_row_to_tmem<Cfg::FMT>(w + c0, w + m0, a_col);
                ptx::tmem_st_wait();
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive(bar_full + 8u * r2.idx);
                    ptx::mbar_arrive(bar_wfree + 8u * r1.idx);   // (behind the stores of what was read from the slot)
                }
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    r1.advance(S1);
                    r2.advance(S2);
                }
            }
            if (!ok) break;
            // Outputs: blocks of 128 rows x 16 tokens, dealt out to the groups; scales fetched ahead of the wait.
            ptx::griddep_wait();   // s_x comes from, and y may still be read by, earlier kernels
            float sx[4];
            const float sw0 = row + lane < R ? __ldg(s_w + (u0 * 8 + row + lane) * sw_stride) : 0.0f;
            const float sw1 = 128 + row + lane < R ? __ldg(s_w + (u0 * 8 + 128 + row + lane) * sw_stride) : 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i) sx[i] = 32 * i + lane < M ? __ldg(s_x + 32 * i + lane) : 0.0f;
            ok = ptx::mbar_wait_warp(bar_acc_full, acc_phase, abort_flag, status_word);
            acc_phase ^= 1u;
            if (!ok) break;
            ptx::tc_fence_after_sync();
            for (int i = g; i < RB * chunks; i += G) {
                const int b = i >= chunks ? 1 : 0, t0 = (i - b * chunks) * 16;
                const int left = R - (b * 128 + row);   // rows of this warp
                if (left <= 0) continue;                // (warp-uniform)
                uint32_t v[16];
                ptx::tmem_ld_32x32b_x16(lanes + (uint32_t)(b * MN + t0), v);
                ptx::tmem_ld_wait_for(v);
                if (cut > 1) {   // partial sums, [token][128 rows]
                    float* mine = partials + (int64_t)t * MN * 128 + row + lane;
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (t0 + j < M) __stcg(mine + (t0 + j) * 128, __uint_as_float(v[j]));
                    continue;
                }
                const float sxv = t0 < 32 ? sx[0] : (t0 < 64 ? sx[1] : (t0 < 96 ? sx[2] : sx[3])), swv = b ? sw1 : sw0;
                const int64_t n = u0 * 8 + b * 128 + row;
                float res[16];
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    res[j] = __uint_as_float(v[j]) * (__shfl_sync(0xFFFFFFFFu, sxv, (t0 & 16) + j) * swv);   // Eq. 4, Eq. 11
                if (!wide) {
                    if (lane < left)
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (t0 + j < M) {
                                if (es == 4)
                                    static_cast<float*>(y)[(int64_t)(t0 + j) * ldy + n + lane] = res[j];
                                else
                                    static_cast<__nv_bfloat16*>(y)[(int64_t)(t0 + j) * ldy + n + lane] = __float2bfloat16_rn(res[j]);
                            }
                    continue;
                }
                // through the warp's staging area, [token][32 rows], from which rows go out in pieces of 16 bytes
                char* yb = static_cast<char*>(y) + ((int64_t)t0 * ldy + n) * es;
                if (es == 2) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(stage + (uint32_t)(j * 64 + lane * 2)),
                                     "h"(__bfloat16_as_ushort(__float2bfloat16_rn(res[j]))) : "memory");
                    __syncwarp();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int tok = h * 8 + (lane >> 2), piece = lane & 3;
                        uint4 o;
                        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(o.x), "=r"(o.y), "=r"(o.z), "=r"(o.w) : "r"(stage + (uint32_t)(tok * 64 + piece * 16)));
                        if (t0 + tok < M && piece * 8 < left) *reinterpret_cast<uint4*>(yb + (int64_t)tok * ldy * 2 + piece * 16) = o;
                    }
                    __syncwarp();
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            asm volatile("st.shared.f32 [%0], %1;" ::"r"(stage + (uint32_t)(j * 128 + lane * 4)), "f"(res[8 * h + j]) : "memory");
                        __syncwarp();
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const int tok = k * 4 + (lane >> 3), piece = lane & 7;
                            uint4 o;
                            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                         : "=r"(o.x), "=r"(o.y), "=r"(o.z), "=r"(o.w) : "r"(stage + (uint32_t)(tok * 128 + piece * 16)));
                            if (t0 + 8 * h + tok < M && piece * 4 < left)
                                *reinterpret_cast<uint4*>(yb + (int64_t)(8 * h + tok) * ldy * 4 + piece * 16) = o;
                        }
                        __syncwarp();
                    }
                }
            }
            if (cut > 1) __threadfence();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_acc_empty);
            ++done_runs;
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(*tmem_slot, Cfg::kTmemCols);
    }
    if (cut > 1 && !*abort_flag) {
        // The CTA that arrives last at its run adds the parts in ascending order, every thread of it with eight loads in
        // flight, and leaves the counter zero.
        const int run = p / cut;
        if (threadIdx.x == 0) {
            __threadfence();
            *ticket = atomicAdd(counters + run, 1u);
        }
        __syncthreads();
        if (*ticket != (uint32_t)(cut - 1)) return;
        ptx::griddep_wait();
        __threadfence();
        const int64_t n0 = first_unit(run) * 8;
        const int R = (int)(first_unit(run + 1) * 8 - n0);
        const float4* parts = reinterpret_cast<const float4*>(partials + (int64_t)run * cut * MN * 128);
        const int step = MN * 32;   // a part further
        const bool whole4 = (ldy & 3) == 0;
        for (int e = (int)threadIdx.x; e < M * 32; e += Cfg::kThreads) {   // four rows of a token each (rows come in eights)
            const int row = (e & 31) * 4, tok = e >> 5;
            if (row >= R) continue;
            const int64_t n = n0 + row;
            const float sx = __ldg(s_x + tok);
            float sw[4], acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int i = 0; i < 4; ++i) sw[i] = __ldg(s_w + (n + i) * sw_stride);
            for (int c0 = 0; c0 < cut; c0 += 8) {   // eight loads in flight
                float4 v[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = c0 + c < cut ? __ldcg(parts + (c0 + c) * step + e) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    acc[0] += v[c].x;
                    acc[1] += v[c].y;
                    acc[2] += v[c].z;
                    acc[3] += v[c].w;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = acc[i] * (sx * sw[i]);   // Eq. 4, Eq. 11
            if (out_dtype == W4A8_OUT_FP32) {
                float* yp = static_cast<float*>(y) + (int64_t)tok * ldy + n;
                if (whole4)
                    *reinterpret_cast<float4*>(yp) = make_float4(acc[0], acc[1], acc[2], acc[3]);
                else
                    for (int i = 0; i < 4; ++i) yp[i] = acc[i];
            } else {
                __nv_bfloat16* yp = static_cast<__nv_bfloat16*>(y) + (int64_t)tok * ldy + n;
                const __nv_bfloat162 lo = __floats2bfloat162_rn(acc[0], acc[1]), hi = __floats2bfloat162_rn(acc[2], acc[3]);
                if (whole4) {
                    *reinterpret_cast<uint2*>(yp) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                } else {
                    yp[0] = lo.x;
                    yp[1] = lo.y;
                    yp[2] = hi.x;
                    yp[3] = hi.y;
                }
            }
        }
        if (threadIdx.x == 0) counters[run] = 0u;
    }
}

}  // namespace w4a8
