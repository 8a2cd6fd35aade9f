// W4A8 linear for more than 128 tokens on CTA pairs: a thread-block cluster of two CTAs works on one tile of
// 256 output channels x 256 H tokens with two-CTA MMAs (tcgen05 cta_group::2), H = 1 or 2.
//
// Bound: long problems run at the power cap, where the work beside the MMAs costs clock; short ones are made of latencies.
// In a pair each CTA expands its own 128 weight rows (the A operand and the accumulator rows of a two-CTA MMA are
// split by rows) and loads half of the activation tile (the B operand is split by tokens), from which both tensor
// cores read.  Per k-block of a 256 x 512 tile (H = 2) a CTA expands 128 rows, writes 16 KB of them and 32 KB of activations
// to shared memory and has 64 KB read by its MMAs, 1024 tensor-pipe cycles; one CTA on its own with a 256 x 256 tile, the
// kernel before this one, expanded 256 rows, wrote 32 + 49 KB and had 96 KB read, which is more than the 128 bytes a
// clock of shared memory allow.  (8192, 28672, 8192): 2011 -> 1500 us back to back (1180-1230 MHz, 1000 W; the library's FP8
// GEMM on FP8 weights 1460), 86-90 % of the tensor pipe at that clock by the cycles of its MMAs; (2048, 4096, 4096): 1130-1170 cycles
// per k-block of the 1024.
//
//   H = 2  both accumulators belong to the tile in flight, expanded weights in shared memory.  The MMAs of a tile's first and
//          last kSkew k-blocks are issued for one accumulator first and then for the other: the second accumulator is
//          drained while the next tile's first MMAs run into the first, the first while the last MMAs run into the second.
//   H = 1  one accumulator and six slots of expanded weights in tensor memory (256 + 192 columns): half the shared-memory
//          traffic of a step, and tiles for problems with few of them.  KP = 2: the two pairs of a cluster of four CTAs take
//          half of K each and exchange half of their partial sums through distributed shared memory, every epilogue warp
//          with the warp of the same rows and columns in the other pair, in pieces of sixteen tokens.
//
// Packed weights go from global memory to registers (a row and k-block per thread), one of a group's stages ahead, and are
// brought to L2 further ahead: a ring of shared memory for them took as long for H = 2 and cost a warp and two barriers.
// (The loads of such a ring must be complete before its slot is released, which program order alone did not ensure.)
// What an arrival orders matters: released at cluster scope, an expanding warp's arrival waited 1500 cycles for
// everything in flight; at CTA scope, with the proxy fence that the operand needs anyway, 180 (a step of H = 2 went
// from 1450 to 1170 cycles, of H = 1 from 960 to 625).
//
// Roles per CTA: warp 0 activation tiles, warp 1 MMA issuer (works in each pair's leader only; both CTAs' warp 1
// allocate and free tensor memory), warps 2-9 epilogue (this CTA's 128 accumulator rows), from warp 10 on G expansion groups
// of four warps (Eq. 10).  One barrier of the leader per stage collects the eight expanding warps' arrivals and both CTAs'
// activation bytes, one commit frees the stage in both CTAs.  No load uses cluster multicast.  Whole tiles; any M, any N (a
// multiple of 16); needs no workspace.  Every wait is bounded.
//
// Epilogue: the accumulator comes out of tensor memory as 16 x 256-bit fragments (a thread holds two neighbouring
// tokens of a channel), is scaled in packed pairs, turned by stmatrix.trans and leaves as 16-byte stores, eight
// channels of a token each: 2 stores per lane and 16 tokens instead of 16.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "w4a8_common.cuh"
#include "w4a8_prefill_plan.h"
#include "w4a8_ptx.cuh"
#include "w4a8_tiled_format.cuh"

namespace w4a8 {

template <int FMT_, int H_, int G_, int S_>
struct PairCfg {
    static constexpr int H = H_;            // accumulators of 256 tokens per tile
    static constexpr int FMT = FMT_;
    static constexpr int kTokens = 256 * H;
    static constexpr int G = G_;            // expansion groups of 4 warps
    static constexpr int S = S_;            // ring of stages: expanded weights and this CTA's half of the activation tile
    static constexpr int kSkew = S - 1;     // k-blocks issued for one accumulator at a time at both ends of a tile (H = 2)
    static constexpr int kAhead = 4;        // of a group's stages, that packed weights are brought to L2 ahead of their load
    static constexpr int kMeta = meta_bytes(FMT);
    static constexpr int kW8Bytes = H == 1 ? 0 : 128 * 128;   // (H = 1: in tensor memory)
    static constexpr bool TS = H == 1;      // expanded weights in tensor memory, behind the accumulator
    static constexpr int kXHalf = 128 * 128;   // this CTA's 128 tokens of one accumulator
    static constexpr int kXBytes = H * kXHalf;
    static constexpr int kOutWarp = 16 * 64 + 512;   // per epilogue warp: 16 tokens x 32 channels, and 128 activation scales
    static constexpr int kOutBytes = 8 * kOutWarp;
    static constexpr int kRecvBytes = H == 1 ? 8 * 8192 : 0;   // partial sums of the pair that takes the other half of K
    static constexpr int kBarBytes = 512;
    static constexpr int kSmemBytes = S * (kXBytes + kW8Bytes) + kRecvBytes + kOutBytes + kBarBytes + 1024;
    static constexpr int kThreads = 32 * (10 + 4 * G);
    // A group handles every G-th stage; with a ring depth that is a multiple of G each slot is always the same group's,
    // so that no wait skips a phase of its barrier (waits tell phases apart by parity only).
    static_assert(S % G == 0, "each ring slot belongs to one expansion group");
    static_assert(kSkew >= 1, "a stage stays free while the skewed MMAs hold theirs");
    static_assert((2 * S + 13) * 8 + 16 <= kBarBytes, "barrier area");
    static_assert(H == 2 || (256 + 32 * S <= 512 && S * kXBytes >= 8 * 8192), "tensor memory columns; room for the partial sums to send");
    static_assert(kSmemBytes <= 232448, "shared memory per CTA");
};

template <class Cfg>
__global__ void __launch_bounds__(Cfg::kThreads)
linear_pair_kernel(const __grid_constant__ CUtensorMap tmap_x,  // X8 u8 [M][K], box 128 x 128, 128B swizzle
                   const uint8_t* __restrict__ wpp, const float* __restrict__ s_x,
                   const float* __restrict__ s_w, int sw_stride, void* __restrict__ y, int64_t ldy, int out_dtype,
                   int M, int N, int K, int TM, int TN, int full_tiles, int KP, unsigned int* status_word) {
    constexpr int H = Cfg::H, G = Cfg::G, S = Cfg::S;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = ptx::smem_addr(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - raw_addr);

    constexpr int kX = S * Cfg::kW8Bytes, kRecv = kX + S * Cfg::kXBytes, kOut = kRecv + Cfg::kRecvBytes, kBars = kOut + Cfg::kOutBytes;
    const uint32_t bars_addr = base + kBars;
    auto bar_full = [&](int s) { return bars_addr + 8u * (uint32_t)s; };                          // leader: stage complete in both CTAs
    auto bar_free = [&](int s) { return bars_addr + 8u * (uint32_t)(S + s); };                    // both: stage consumed
    auto bar_acc_full = [&](int b) { return bars_addr + 8u * (uint32_t)(2 * S + b); };            // both
    auto bar_acc_empty = [&](int b) { return bars_addr + 8u * (uint32_t)(2 * S + 2 + b); };       // leader
    const uint32_t bar_drain = bars_addr + 8u * (uint32_t)(2 * S + 4);
    auto bar_red = [&](int w) { return bars_addr + 8u * (uint32_t)(2 * S + 5 + w); };             // local: partial sums for epilogue warp w landed
    constexpr int kNumBars = 2 * S + 13;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + kBars + 8 * kNumBars);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    auto stage_w8 = [&](int s) { return base + (uint32_t)(s * Cfg::kW8Bytes); };
    auto stage_x = [&](int s) { return base + (uint32_t)(kX + s * Cfg::kXBytes); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t ctarank = ptx::cluster_ctarank(), pair_leader = ctarank & ~1u;
    const uint32_t rank = ctarank & 1u;   // within the pair
    const bool leader = rank == 0;
    const uint16_t pair_mask = (uint16_t)(3u << pair_leader);
    const int KBall = K >> 7;
    // this pair's share of K (KP = 1: all of it; KP = 2: the two pairs of a cluster of four CTAs take half each)
    const int kp = (int)(ctarank >> 1);
    const int kb0 = KP == 1 ? 0 : kp * KBall / KP, KB = KP == 1 ? KBall : (kp + 1) * KBall / KP - kb0;
    const uint8_t* meta_base = wpp + (int64_t)KBall * N * kRowCodeBytes;
    const int C = (int)gridDim.x / (2 * KP), c = (int)blockIdx.x / (2 * KP);
    const int Tt = TM * TN;
    const int n_tiles = c < Tt ? (Tt - c + C - 1) / C : 0;  // tiles c, c + C, ...
    const int n_it = n_tiles * KB;
    // accumulators of 256 tokens that a token tile needs
    auto halves_of = [&](int mt) { return H == 2 && M - mt * Cfg::kTokens > 256 ? 2 : 1; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            ptx::mbar_init(bar_full(s), 8 + 1);   // four expanding warps of each CTA, the activation tiles' request
            ptx::mbar_init(bar_free(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(bar_acc_full(b), 1);
            ptx::mbar_init(bar_acc_empty(b), 16);   // eight epilogue warps of each CTA
        }
        ptx::mbar_init(bar_drain, 1);
        for (int w = 0; w < 8; ++w) ptx::mbar_init(bar_red(w), 1);
        *abort_flag = 0u;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_x);
    }
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), 512);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync_all();  // the peer's barriers exist before anything arrives on them
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    ptx::griddep_launch_dependents();

    if (warp == 0) {
        // ------------------------------------------------------------------ activation tiles
        bool ok = true;
        ptx::Ring r;
        int issued = 0, nt, mt = 0;
        if (n_tiles > 0) pair_tile(c, full_tiles, TN, nt, mt);   // (ahead of the wait: nothing is between it and the first request)
        ptx::griddep_wait();
        for (int j = 0; j < n_tiles && ok; ++j) {
            if (j > 0) pair_tile(c + j * C, full_tiles, TN, nt, mt);
            const int halves = halves_of(mt);
            const int y0 = mt * Cfg::kTokens + (int)rank * 128;
            for (int kb = 0; kb < KB; ++kb) {
                if (issued >= S) ok = ptx::mbar_wait_warp(bar_free(r.idx), r.phase ^ 1u, abort_flag, status_word);
                if (!ok) break;
                const uint32_t full = bar_full(r.idx), full_leader = ptx::map_to_cta(full, pair_leader), dst = stage_x(r.idx);
                if (ptx::elect_one()) {
                    if (leader) ptx::mbar_arrive_expect_tx(full, (uint32_t)(2 * halves * Cfg::kXHalf));
                    ptx::tma_load_2d_pair(dst, &tmap_x, (kb0 + kb) * 128, y0, full_leader);
                    if (H == 2 && halves == 2) ptx::tma_load_2d_pair(dst + (uint32_t)Cfg::kXHalf, &tmap_x, (kb0 + kb) * 128, y0 + 256, full_leader);
                }
                r.advance(S);
                ++issued;
            }
        }
        if (!ok && leader && lane == 0) {
            // Gave up: let both CTAs' copies already in flight land (the peer leaves behind the cluster barrier below).
            // The barriers count the expanding warps as well, which may have given up too: a part of the limit only.
            const uint64_t t0 = ptx::globaltimer_ns();
            for (int it = issued > S ? issued - S : 0; it < issued; ++it)
                while (!ptx::mbar_try_wait(bar_full(it % S), (uint32_t)((it / S) & 1)) &&
                       ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs / 20) {
                }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader only)
        if (leader) {
            constexpr uint32_t idesc = ptx::umma_idesc_e4m3_f32(256, 256);
            bool ok = true;
            ptx::Ring r;         // next stage
            bool ready = false;  // ... is known to be complete
            int left = n_it;     // stages not yet begun
            // The queue of MMAs is short: a wait between two stages, a hundred cycles even where the stage has long been
            // complete, left the tensor pipe idle for as long.  The next stage is therefore looked at while a part of
            // this one's MMAs is still to be issued.
            auto peek = [&]() {
                if (left > 0) ready = __all_sync(0xFFFFFFFFu, ptx::mbar_test_wait(bar_full(r.idx), r.phase)) != 0;
            };
            auto wait_stage = [&]() -> bool {
                const bool got = ready || ptx::mbar_wait_warp(bar_full(r.idx), r.phase, abort_flag, status_word);
                ready = false;
                --left;
                ptx::tc_fence_after_sync();
                return got;
            };
            int used1 = 0;   // H = 2: tiles so far that used the second accumulator
            for (int j = 0; j < n_tiles && ok; ++j) {
                int nt, mt;
                pair_tile(c + j * C, full_tiles, TN, nt, mt);
                const int halves = halves_of(mt);
                if (j >= 1) {
                    ok = ptx::mbar_wait_warp(bar_acc_empty(0), (uint32_t)((j - 1) & 1), abort_flag, status_word);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                }
                const uint32_t acc0 = tmem_base, acc1 = tmem_base + 256u;
                if (H == 1 || halves == 1) {
                    for (int i = 0; i < KB; ++i) {
                        ok = wait_stage();
                        if (!ok) break;
                        const uint32_t a_lo = Cfg::TS ? tmem_base + (uint32_t)(256 + 32 * r.idx) : ptx::umma_desc_lo(stage_w8(r.idx));
                        const uint32_t b_lo = ptx::umma_desc_lo(stage_x(r.idx)), fr = bar_free(r.idx);
                        r.advance(S);
                        if (ptx::elect_one()) {
                            if (Cfg::TS) ptx::umma_f8_kblock_pair_ts(acc0, a_lo, b_lo, idesc, (uint32_t)i);
                            else ptx::umma_f8_kblock_pair(acc0, a_lo, b_lo, idesc, (uint32_t)i);
                            if (left >= S) ptx::umma_commit_pair(fr, pair_mask);   // (the slot is used again: see the closing barrier)
                        }
                    }
                    if (ok && ptx::elect_one()) ptx::umma_commit_pair(bar_acc_full(0), pair_mask);
                } else {
                    bool free1 = used1 == 0;   // second accumulator known to be drained
                    int i = 0;
                    while (i < KB) {
                        // d stages' MMAs into the first accumulator, then the same stages' into the second
                        int d = 1;
                        if (i == 0 && !free1) d = KB < Cfg::kSkew ? KB : Cfg::kSkew;
                        else if (KB - i <= Cfg::kSkew) d = KB - i;
                        const bool last = i + d == KB;
                        ptx::Ring r1 = r;
                        for (int k = 0; k < d; ++k) {
                            ok = wait_stage();
                            if (!ok) break;
                            const uint32_t a_lo = ptx::umma_desc_lo(stage_w8(r.idx)), b_lo = ptx::umma_desc_lo(stage_x(r.idx));
                            r.advance(S);
                            if (ptx::elect_one()) ptx::umma_f8_kblock_pair(acc0, a_lo, b_lo, idesc, (uint32_t)(i + k));
                            peek();
                        }
                        if (!ok) break;
                        if (last && ptx::elect_one()) ptx::umma_commit_pair(bar_acc_full(0), pair_mask);
                        if (!free1) {
                            ok = ptx::mbar_wait_warp(bar_acc_empty(1), (uint32_t)((used1 - 1) & 1), abort_flag, status_word);
                            if (!ok) break;
                            ptx::tc_fence_after_sync();
                            free1 = true;
                        }
                        for (int k = 0; k < d; ++k) {
                            const bool again = left + (d - 1 - k) >= S;   // the slot is used again
                            const uint32_t a_lo = ptx::umma_desc_lo(stage_w8(r1.idx));
                            const uint32_t b_lo = ptx::umma_desc_lo(stage_x(r1.idx) + (uint32_t)Cfg::kXHalf);
                            const uint32_t fr = bar_free(r1.idx);
                            if (ptx::elect_one()) {
                                ptx::umma_f8_kblock_pair(acc1, a_lo, b_lo, idesc, (uint32_t)(i + k));
                                if (again) ptx::umma_commit_pair(fr, pair_mask);
                            }
                            r1.advance(S);
                        }
                        if (last && ptx::elect_one()) ptx::umma_commit_pair(bar_acc_full(1), pair_mask);
                        i += d;
                    }
                    ++used1;
                }
            }
            if (!ok && lane == 0) {
                // Gave up: let the MMAs already issued finish before tensor memory is freed.
                ptx::umma_commit_pair(bar_drain, (uint16_t)(1u << pair_leader));
                const uint64_t t0 = ptx::globaltimer_ns();
                while (!ptx::mbar_try_wait(bar_drain, 0u) && ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs) {
                }
            }
        }
        __syncwarp();
    } else if (warp < 10) {
        // ------------------------------------------------------------------ epilogue (8 warps)
        // This CTA's accumulator rows: lane = output channel, column = token.  Two warps share a lane quarter, each
        // takes 128 of an accumulator's 256 tokens.
        const int q = warp & 3, side = (warp - 2) >> 2;
        const uint32_t out_s = base + (uint32_t)(kOut + (warp - 2) * Cfg::kOutWarp), sx_s = out_s + 1024u;
        const bool vec_ok = out_dtype != W4A8_OUT_FP32 && (ldy & 7) == 0;   // (the base is 16-byte aligned)
        bool ok = true;
        int used1 = 0;   // H = 2: tiles so far that used the second accumulator
        const int last1 = c < full_tiles * TN ? (full_tiles * TN - c + C - 1) / C - 1 : -1;   // H = 2: last tile that uses it
        ptx::griddep_wait();  // scales come from, outputs may still be in use by, earlier kernels
        for (int j = 0; j < n_tiles && ok; ++j) {
            int nt, mt;
            pair_tile(c + j * C, full_tiles, TN, nt, mt);
            const int halves = halves_of(mt);
            const int n0 = nt * 256 + (int)rank * 128 + q * 32;   // this warp's first channel
            // Eq. 11 scales: of the fragment's channels (rows lane / 4 + 8 g), or of this lane's channel
            float swn[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int n = n0 + (vec_ok ? (lane >> 2) + 8 * g : lane);
                swn[g] = n < N ? __ldg(s_w + (int64_t)n * sw_stride) : 0.0f;
            }
#pragma unroll 1
            for (int h = 0; h < halves; ++h) {
                // this warp's columns of the accumulator (K cut in two: half of them, the other pair takes the others)
                const int cols = KP == 1 ? 128 : 64, first = KP == 1 ? side * 128 : kp * 128 + side * 64;
                const int m0 = mt * Cfg::kTokens + h * 256 + first;
                // Eq. 4 scales of the warp's tokens
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int m = m0 + 32 * k + lane;
                    const float v = 32 * k < cols && m < M ? __ldg(s_x + m) : 0.0f;
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(sx_s + (uint32_t)(4 * (32 * k + lane))), "f"(v) : "memory");
                }
                __syncwarp();
                if (KP == 2 && lane == 0) ptx::mbar_arrive_expect_tx(bar_red(warp - 2), 8192u);
                const int use = h == 0 ? j : used1++;
                ok = ptx::mbar_wait_warp(bar_acc_full(h), (uint32_t)(use & 1), abort_flag, status_word);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t acc_q = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * 256);
                const int valid = M - m0 < cols ? M - m0 : cols;   // tokens of this warp inside the problem
                // sixteen tokens of the warp's 32 channels: as fragments, or a lane = a channel
                auto fetch = [&](uint32_t (&v)[16], int col) {
                    if (vec_ok) {
                        ptx::tmem_ld_16x256b_x2(acc_q + (uint32_t)col, v);
                        ptx::tmem_ld_16x256b_x2(acc_q + (16u << 16) + (uint32_t)col, v + 8);
                    } else {
                        ptx::tmem_ld_32x32b_x16(acc_q + (uint32_t)col, v);
                    }
                };
                const uint32_t recv = base + (uint32_t)(kRecv + (warp - 2) * 8192 + lane * 16);
                if (Cfg::TS && KP == 2) {
                    // The other pair's columns go to the CTA of that pair with the same rows, as they come out of tensor
                    // memory: through this CTA's activation ring, which is idle (the tile's MMAs have completed).
                    const uint32_t send = base + (uint32_t)(kX + (warp - 2) * 8192);
                    const uint32_t there = ptx::map_to_cta(base + (uint32_t)(kRecv + (warp - 2) * 8192), ctarank ^ 2u);
                    const uint32_t there_bar = ptx::map_to_cta(bar_red(warp - 2), ctarank ^ 2u);
#pragma unroll 1
                    for (int ch = 0; ch < 4; ++ch) {
                        uint32_t v[16];
                        fetch(v, (1 - kp) * 128 + side * 64 + 16 * ch);
                        ptx::tmem_ld_wait_for(v);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            ptx::st_shared_v4(send + (uint32_t)((ch * 4 + i) * 512 + lane * 16),
                                              make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
                        ptx::fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) ptx::bulk_copy_to_cta(there + (uint32_t)(ch * 2048), send + (uint32_t)(ch * 2048), 2048u, there_bar);
                        __syncwarp();
                    }
                    ok = ptx::mbar_wait_warp(bar_red(warp - 2), 0u, abort_flag, status_word);   // (one tile per cluster)
                    if (!ok) break;
                }
                // the other pair's partial sums (a sum of two terms does not depend on their order)
                auto add_recv = [&](uint32_t (&v)[16], int c0) {
                    if (Cfg::TS && KP == 2) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float4 t;
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                         : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w)
                                         : "r"(recv + (uint32_t)((c0 * 4 / 16 + i) * 512)));
                            v[4 * i] = __float_as_uint(__uint_as_float(v[4 * i]) + t.x);
                            v[4 * i + 1] = __float_as_uint(__uint_as_float(v[4 * i + 1]) + t.y);
                            v[4 * i + 2] = __float_as_uint(__uint_as_float(v[4 * i + 2]) + t.z);
                            v[4 * i + 3] = __float_as_uint(__uint_as_float(v[4 * i + 3]) + t.w);
                        }
                    }
                };
                if (vec_ok) {
                    __nv_bfloat16* yb = reinterpret_cast<__nv_bfloat16*>(y);
                    const int ch = n0 + 8 * (lane & 3);          // the eight channels of this lane's stores
                    // matrix i of a store to shared memory = channels 8 i .. 8 i + 7, row = token; 16-byte pieces permuted
                    // so that the eight rows of a matrix fall into different banks
                    const uint32_t st_a = out_s + (uint32_t)((lane & 7) * 64 + ((((lane >> 3) ^ (lane >> 1)) & 3) << 4));
                    const uint32_t ld_a = out_s + (uint32_t)((lane >> 2) * 64 + (((lane ^ (lane >> 3)) & 3) << 4));
                    uint32_t va[16], vb[16];
                    auto put = [&](uint32_t (&v)[16], int c0) {
                        add_recv(v, c0);
#pragma unroll
                        for (int tg = 0; tg < 2; ++tg) {
                            float sx0, sx1;
                            asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];"
                                         : "=f"(sx0), "=f"(sx1)
                                         : "r"(sx_s + (uint32_t)(4 * (c0 + 8 * tg + 2 * (lane & 3)))));
                            uint32_t o[4];
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                float a0, a1, r0, r1;
                                ptx::mul_f32x2(sx0, sx1, swn[g], swn[g], a0, a1);
                                const int at = 8 * (g >> 1) + 4 * tg + 2 * (g & 1);
                                ptx::mul_f32x2(__uint_as_float(v[at]), __uint_as_float(v[at + 1]), a0, a1, r0, r1);
                                const __nv_bfloat162 p = __floats2bfloat162_rn(r0, r1);
                                o[g] = *reinterpret_cast<const uint32_t*>(&p);
                            }
                            ptx::stmatrix_x4_trans(st_a + (uint32_t)(tg * 512), o);
                        }
                        __syncwarp();
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            const int t = c0 + 8 * p + (lane >> 2);
                            uint4 o;
                            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                         : "=r"(o.x), "=r"(o.y), "=r"(o.z), "=r"(o.w)
                                         : "r"(ld_a + (uint32_t)(p * 512))
                                         : "memory");
                            if (t < valid && ch < N) *reinterpret_cast<uint4*>(yb + (int64_t)(m0 + t) * ldy + ch) = o;
                        }
                        __syncwarp();
                    };
                    fetch(va, first);
#pragma unroll 1
                    for (int c0 = 0; c0 < cols; c0 += 32) {
                        // (the next sixteen tokens are on their way while these are scaled and stored)
                        if (c0 >= valid) break;   // warp-uniform
                        ptx::tmem_ld_wait_for(va);
                        fetch(vb, first + c0 + 16);
                        put(va, c0);
                        ptx::tmem_ld_wait_for(vb);
                        if (c0 + 32 < cols) fetch(va, first + c0 + 32);
                        put(vb, c0 + 16);
                    }
                    ptx::tmem_ld_wait();
                } else {
                    const int n = n0 + lane;
#pragma unroll 1
                    for (int c0 = 0; c0 < cols; c0 += 16) {
                        if (c0 >= valid) break;   // warp-uniform
                        uint32_t v[16];
                        fetch(v, first + c0);
                        ptx::tmem_ld_wait_for(v);
                        add_recv(v, c0);
                        if (n < N) {
#pragma unroll
                            for (int jj = 0; jj < 16; ++jj) {
                                if (c0 + jj >= valid) break;
                                float sx;
                                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(sx) : "r"(sx_s + (uint32_t)(4 * (c0 + jj))));
                                const float res = __uint_as_float(v[jj]) * (sx * swn[0]);
                                const int64_t at = (int64_t)(m0 + c0 + jj) * ldy + n;
                                if (out_dtype == W4A8_OUT_FP32) reinterpret_cast<float*>(y)[at] = res;
                                else reinterpret_cast<__nv_bfloat16*>(y)[at] = __float2bfloat16_rn(res);
                            }
                        }
                    }
                }
                ptx::tc_fence_before_sync();
                __syncwarp();
                // (a later tile uses the accumulator: see the closing barrier)
                if (lane == 0 && j < (h == 0 ? n_tiles - 1 : last1)) ptx::mbar_arrive_cluster(ptx::map_to_cta(bar_acc_empty(h), pair_leader));
            }
        }
    } else {
        // ------------------------------------------------------------------ expansion groups
        const int g = (warp - 10) >> 2;
        const int r = (warp & 3) * 32 + lane;   // (a warp reaches the tensor-memory lanes of its quarter)
        // Codes and meta word of row r of this CTA's half of the tile (a row past the last channel repeats the last one: its
        // sums are not stored) are loaded one of the group's stages ahead, which covers the latency of L2, and brought to L2
        // kAhead stages ahead of that, by sixteen lanes for the codes of the warp's 32 rows and one for their meta data.
        // Weights depend on no earlier kernel.
        struct At {
            int j, kb, n0;
        };
        auto go = [&](At& at, int step) {
            at.kb += step;
            while (at.kb >= KB && KB > 0) {
                at.kb -= KB;
                if (++at.j < n_tiles) {
                    int nt, mt;
                    pair_tile(c + at.j * C, full_tiles, TN, nt, mt);
                    at.n0 = nt * 256 + (int)rank * 128;
                }
            }
        };
        At cur = {-1, g + KB, 0}, far = cur;   // (k-block g of tile 0, once go() has been there)
        uint32_t pk[16], mbits = 0u;
        auto fetch = [&]() {
            const int n = cur.n0 + r < N ? cur.n0 + r : N - 1;
            const int64_t row = (int64_t)(kb0 + cur.kb) * N + n;
            load_row_codes_global(wpp + (row - (n & 7)) * kRowCodeBytes + (n & 7) * 16, pk);
            mbits = load_meta_word_global<Cfg::FMT>(meta_base + row * Cfg::kMeta);
        };
        auto prefetch = [&]() {
            const int n = far.n0 + (warp & 3) * 32;
            const int64_t row = (int64_t)(kb0 + far.kb) * N + n;
            if (far.j < n_tiles && lane <= 16 && n + 2 * lane < N) {
                const uint8_t* line = lane < 16 ? wpp + row * kRowCodeBytes + lane * 128 : meta_base + row * Cfg::kMeta;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
            }
        };
        go(cur, 0);
        far = cur;
        for (int i = 0; i < Cfg::kAhead; ++i) {
            go(far, G);
            prefetch();
        }
        if (g < n_it) fetch();
        for (int it = g; it < n_it; it += G) {
            const int s = it % S;
            if (it >= S && !ptx::mbar_wait_warp(bar_free(s), (uint32_t)((it / S - 1) & 1), abort_flag, status_word)) break;
            uint32_t now[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) now[i] = pk[i];
            const uint32_t m = mbits;
            if (it + G < n_it) {
                go(cur, G);
                fetch();
                go(far, G);
                prefetch();
            }
            if constexpr (Cfg::TS) {
                ptx::tc_fence_after_sync();
                expand_row_to_tmem<Cfg::FMT, true>(now, m, tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(256 + 32 * s));
                ptx::tmem_st_wait();
                ptx::tc_fence_before_sync();
            } else {
                expand_row_to_smem<Cfg::FMT, true>(now, m, r, stage_w8(s) + (uint32_t)r * 128u);
                ptx::fence_proxy_async_smem();
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(bar_full(s), pair_leader));
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    // Closing barrier: no CTA of the cluster leaves while another may still reach into its shared memory or barriers.  It
    // orders execution only (a releasing arrival would first wait for this thread's output stores), so nothing may be sent to
    // another CTA that no thread of that CTA has waited for by now:
    //   stage complete (leader: the peer's expanding warps, both CTAs' activation tiles)   by the issuer, before the stage's MMAs
    //   stage free (both: the leader's commits)               by the warps that fill the slot again; not sent for the last S stages
    //   accumulator complete (both: the leader's commits)     by the epilogue warps
    //   accumulator drained (leader: the peer's epilogue warps)   by the issuer, before the next tile in it; not sent after the last
    //   partial sums (KP = 2: the other pair's copies)        by the epilogue warps
    // (Sent always and waited for behind the loops, (2048, 4096, 4096) took 29.3 us in place of 28.6, (8192, 28672, 8192) 1332 in place of 1301.)
    const bool gave_up = *abort_flag != 0u;   // (the same for all threads: nobody of this CTA waits any more)
    if (gave_up) ptx::cluster_arrive();
    else ptx::cluster_arrive_relaxed();
    ptx::cluster_wait();
    if (gave_up) {
        // Not all of it has been waited for: partial sums that the other pair has sent all the same land before this CTA's
        // shared memory goes away, and a late arrival of a CTA that has not given up has 2 ms.
        const uint64_t t0 = ptx::globaltimer_ns();
        if (Cfg::TS && KP == 2 && threadIdx.x < 8)
            while (!ptx::mbar_try_wait(bar_red((int)threadIdx.x), 0u) && ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs / 20) {
            }
        while (ptx::globaltimer_ns() - t0 < ptx::kWaitLimitNs / 1000) {
        }
    }
    __syncwarp();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 512);
    }
}

}  // namespace w4a8
