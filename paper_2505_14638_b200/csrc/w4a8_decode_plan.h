// Up to 128 tokens on prepacked layers (and up to sixteen on canonical ones): which kernel runs and with which plan.  Host code
// without CUDA, so that a host test can ask for the route of a shape.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "../../include/w4a8.h"
#include "w4a8_prefill_plan.h"

namespace w4a8 {

constexpr int kFmtCanonical = W4A8_FMT_CANONICAL;
constexpr int kFmtTiled = W4A8_FMT_TILED;
constexpr int kFmtTiledSignMag = W4A8_FMT_TILED_SIGNMAG;
constexpr int kFmtTiledFp8 = W4A8_FMT_TILED_FP8;   // FP8 weights (W8A8 comparison scheme): 128 bytes per row and k-block, no meta data

constexpr int kRowCodeBytes = 64;  // one row of one k-block: 128 INT4 codes
W4A8_HOST_DEVICE constexpr int meta_bytes(int fmt) {
    return fmt == kFmtTiledSignMag ? 2 : (fmt == kFmtTiled ? 4 : 0);   // (FP8: none; canonical: in arrays of their own)
}

constexpr int64_t kHostFewOutputs = 40000;   // outputs in host memory up to which the kernels for small layers write them
constexpr int kRowsMaxM = 128;    // token counts served by linear_rows_kernel (and what runs beside it up to there)

// Launch-time plan of linear_direct_kernel.
struct DirPlan {
    int P;    // CTAs; CTA p takes units [p NU / P, (p + 1) NU / P)
    int Wq;   // warps that share a row tile's k-block quads
    int Tc;   // row tiles in progress at once (Wq * Tc <= 16)
    int xpitch;   // bytes between two tokens in shared memory
};

// ... and of linear_rows_kernel.
struct RowsPlan {
    int T;       // runs of rows x parts of K; CTA p takes tiles p, p + gridDim.x, ... (cut: one tile each)
    int cut;     // parts of K (1: none; above, the partial sums meet in the workspace)
    int units, more;   // units of eight rows in a run; the first `more` runs have one more
    int RB;      // blocks of 128 rows in a run (1 or 2)
    int MN;      // tokens rounded up to sixteen
    int S1;      // ring of packed stages
    int S2;      // ring of expanded stages and their activation tiles
    int whalf;   // bytes of a k-block in a slot of the first
    int smem;
};
// What a CTA of it has room for.
template <int FMT_, bool HALF_ = false>
struct RowsSizes {
    static constexpr int G = HALF_ ? 2 : 4;     // expansion groups
    static constexpr int kMeta = meta_bytes(FMT_);
    static constexpr int kS1Max = 16, kS2Max = 8;
    static constexpr int kTmemCols = HALF_ ? 256 : 512;
    static constexpr int kStageBytes = 1024;                    // per warp: 16 tokens x 32 rows of outputs (FP32: 8 tokens)
    static constexpr int kOutBytes = 4 * G * kStageBytes;
    static constexpr int kBarBytes = 512;
    static constexpr int kSmemBudget = (HALF_ ? 110 : 224) * 1024;
    static constexpr int kFixed = kOutBytes + kBarBytes + 1024;
    static_assert((2 * kS1Max + 2 * kS2Max + 3) * 8 + 16 <= kBarBytes, "barrier area");
};

// Up to 128 tokens: whole tiles of the persistent kernel, at most one per SM, where K is so short that start and end of a launch
// count more than its main loop: its roles are fewer and set up faster than linear_rows_kernel's, nothing is exchanged, no cluster
// has to be placed.  Time, quantization and linear layer back to back, weights not in L2, this / linear_rows_kernel / the other
// candidate (up to sixteen tokens linear_direct_kernel, above K cut in clusters), us:
//   M <= 8   (8064, 256) 4.0 / 4.4 / 4.2, (992, 640) 4.4 / 4.6 / -, (672, 1792) 6.0 / 7.0 / -, (8656, 2560) 7.9 / 8.5 / 8.9
//   M <= 16  (4672, 896) 4.8 / 5.5 / 5.9, (5312, 1408) 5.4 / 7.2 / 6.5, (8048, 2176) 6.9 / 8.5 / 10.0, (1344, 3456) 9.3 / 7.4 / 7.6
//   above    (57, 11776, 640) 5.3 / 5.8 / -, (126, 7360, 512) 5.6 / 6.2 / 9.6, (46, 7872, 1024) 5.4 / 5.7 / 7.1, (29, 800, 1920) 6.4 / 6.8 / 5.5
// The limits follow 1050 shapes of up to 16 tokens and 560 of 17..128, timed that way and as linear layers alone, back to back, as a
// caller has it that runs several on one X8.  With more tiles than half the SMs linear_rows_kernel fills all SMs as well: there
// K up to 512 for so many tiles (up to sixteen tokens; CTAs of half an SM above, us with quantization, alone: (8, 14384, 512) 4.7, 4.2
// here and 4.6, 3.5 there, (6, 11104, 512) 4.3, 3.6 and 4.5, 3.1, (12, 18128, 256) 4.2, 3.7 and 4.2, 2.8), or K up to 1024, above 32 tokens
// 2432 or 3072 ((106, 9616, 2176) 8.6, 7.4 and 8.6, 8.2; with zero-points (101, 16080, 2304) 9.7, 8.7 and 10.3, 9.8).  More tiles than
// SMs: two k-blocks with zero-points ((108, 24032, 256) 6.9, 6.6 and 7.4, 6.8), and where a run of rows would exceed 256 and a second round comes to be all
// but empty ((124, 39040, 1024) 14.1, 11.8 and 15.9, 15.3).
// Outputs in host memory: always where there are more tiles than half the SMs and more than sixteen tokens; the bus takes its
// stores better, (77, 28672, 4096) 119 us host to host against 128.  Up to sixteen tokens not for more than kHostFewOutputs, like
// linear_direct_kernel.
inline bool whole_tiles_apply(int64_t M, int64_t N, int64_t K, int fmt, int sms, bool y_on_host) {
    const int64_t tiles = (N + 127) / 128;
    const bool sm = fmt == kFmtTiledSignMag;
    if (y_on_host && M <= 16 && M * N > kHostFewOutputs) return false;
    if (2 * tiles > sms) {
        if (M <= 16) return K <= 512 && 20 * tiles <= sms * (K > 384 ? 14 : 17);
        if (y_on_host) return true;
        if (tiles > sms) return N > (int64_t)256 * sms ? K <= 2048 : !sm && K <= 256 && 2 * tiles <= 3 * sms;
        return K <= (M <= 32 ? 1024 : (sm ? 2432 : 3072));
    }
    if (M > 16) return 100 * (K / 128) <= 800 + 12 * M;
    return K <= (N < 1024 ? 2304 : (sm ? 2944 : 2688));
}

// 17..128 tokens: whether cutting the tiles' K between the CTAs of clusters of `cl` pays for the exchange of the partial sums: the
// k-blocks that a CTA is spared against what grows with the tokens.  Fitted to 400 shapes of up to 9472 channels;
// against linear_rows_kernel, us: (124, 7328, 512) 10.0 / 6.7, (112, 5600, 3584) 12.3 / 10.2, (20, 4096, 4096) 7.5 / 9.7, (20, 4096,
// 14336) 12.6 / 24.9.
inline bool cluster_kcut_pays(int64_t M, int64_t K, int cl) { return 50 * (K / 128) * (cl - 1) >= cl * (120 + 7 * M); }

// Few tiles (at most half as many 128-row tiles as SMs) and at most 128 tokens: CTAs per tile of the plan
// that cuts K between the CTAs of a thread-block cluster (0: the plan does not apply).  Every CTA keeps
// at least two k-blocks.
inline int cluster_kcut_ctas(int64_t M, int64_t N, int64_t K, int sms) {
    if (M > 128) return 0;
    const int64_t TN = (N + 127) / 128, KB = K / 128;
    int64_t c = sms / TN;
    if (c > 8) c = 8;
    while (c > 1 && KB < 2 * c) --c;
    return c >= 2 ? (int)c : 0;
}

constexpr int kDirMaxSmem = 227 * 1024;

inline int64_t direct_xpitch(int64_t K) { return (K / 128 * 144 + 64 + 127) / 128 * 128 + 64; }

inline size_t direct_smem(int64_t M, int64_t K, int nt) {
    return (size_t)M * (size_t)direct_xpitch(K) + (size_t)((M + 3) & ~(int64_t)3) * 4 + (size_t)2 * 16 * 8 * nt * 20 * 4;
}

// Arrangement of the sixteen warps of a CTA with the fewest rounds (units of work per warp); returns those.
inline int64_t make_direct_plan(int64_t N, int64_t K, int sms, DirPlan* plan) {
    const int64_t NU = N / 8;
    plan->P = (int)(sms < NU ? sms : NU);
    plan->xpitch = (int)direct_xpitch(K);
    const int64_t T = ((NU + plan->P - 1) / plan->P + 1) / 2, Q = (K / 128 + 3) / 4;
    int64_t best = INT64_MAX;
    for (int wq = 1; wq <= 16 && wq <= Q; ++wq) {
        const int64_t tc = 16 / wq, rounds = ((T + tc - 1) / tc) * ((Q + wq - 1) / wq);
        if (rounds < best) {
            best = rounds;
            plan->Wq = wq;
            plan->Tc = (int)tc;
        }
    }
    return best;
}

// Layers at up to sixteen tokens for which linear_direct_kernel is the faster one: those of few weights, where its short start and
// end count; its expansion does not keep up with larger ones (the FP8 fragments of its MMA are converted to 16 bits on the pipe that
// expands), and a short K is better walked by one CTA per tile (whole_tiles_apply, with the same shapes).  Time, quantization
// and linear layer back to back, weights not in L2, this kernel / whole tiles / linear_rows_kernel, us:
//   M <= 8   (1616, 512) 4.1 / 4.1 / 4.5, (1104, 1408) 4.4 / 5.4 / 7.1, (2160, 3328) 5.2 / 9.0 / 6.9, (7488, 2048) 7.5 / 6.7 / 7.7,
//            (5968, 3968) 8.8 / 9.3 / 8.1, (4960, 8192) 15.4 / 20.0 / 11.2
//   M <= 16  (2752, 512) 5.4 / 4.1 / 4.7, (1072, 1920) 5.3 / 6.4 / 7.5, (3472, 1280) 6.1 / 5.2 / 6.9, (2352, 8064) 10.9 / 19.8 / 9.0
// (Up to 2.2 million weights from nine tokens on: launched one by one such a layer is bound by the host's calls, of which the tensor map
// of the other kernels takes 0.3 us: (16, 1024, 1024) 5.8 against 6.1 us; replayed from a graph it takes 5.3 against 4.8.)
// And layers of which every warp has one unit of work, up to four tokens with a longer K, nine to twelve of up to 4 million weights
// (with quantization, alone; this / linear_rows_kernel with CTAs of half an SM): (1, 2048, 7168) 7.0, 5.4 / 7.6, 6.4, (4, 3888, 3456) 7.0, 5.3 / 7.3,
// 5.8, (1, 4096, 4096) 7.3, 6.0 / 7.5, 5.9; (12, 2304, 1664) 5.4, 3.5 / whole tiles 5.8, 4.3.
// Layers of more 128-channel tiles than half the SMs keep the kernels that walk all of K in one chain of MMAs: a chain launch gives
// the same bits there, and this one is the slower by (14352, 512) 4.6 / 4.6 to (16640, 512) 6.3 / 4.9.
// Canonical, against the kernel of one tile per CTA: M = 8 (1024, 1024) 0.46, (6144, 4096) 0.87, (12288, 2048) 0.81; M = 16 (6144,
// 4096) 0.98, (2048, 8192) 1.05; (1552, 14336) M = 4 1.01, M = 8 1.05, M = 9 1.15; (4096, 6144) M = 12 1.06.  24 tokens: level at
// (1024, 1024), slower everywhere else.
inline bool direct_applies(int64_t M, int64_t N, int64_t K, int fmt, int sms, DirPlan* plan) {
    if (M > 16 || N < 1024 || direct_smem(M, K, M <= 8 ? 1 : 2) > (size_t)kDirMaxSmem) return false;
    const int64_t rounds = make_direct_plan(N, K, sms, plan), weights = N * K;
    const bool few = M <= 8;
    if (fmt == kFmtCanonical)
        return rounds <= 2 && weights <= (few || K <= 4096 || K > 8192 ? 26 : 16) * (int64_t)1000000 && (K <= 11008 || M <= 4);
    if (2 * ((N + 127) / 128) > sms) return false;
    if (rounds == 1 && (M <= 4 ? K >= 2304 : (M > 8 && M <= 12 && K >= 1408 && weights <= 4000000))) return true;
    const bool sm = fmt == kFmtTiledSignMag;
    return few ? weights <= 8000 * K - (sm ? 2000000 : 3000000) && weights <= (sm ? 12000000 : 10000000)
               : K >= 1024 && weights <= 8000000 && (weights <= 5000 * K - 5000000 || weights <= 2200000);
}

// Up to 128 tokens: the plan of linear_rows_kernel.  K is cut (may_cut: up to sixteen tokens, with a workspace) where the
// channels make less than half as many runs of 128 rows as there are SMs.
inline int64_t rows_cut(int64_t N, int64_t K, int sms, bool may_cut) {
    const int64_t blocks = (N + 127) / 128;
    if (!may_cut || blocks * 2 > sms) return 1;
    int64_t cut = sms / blocks;
    if (cut > K / 512) cut = K / 512;   // at least four k-blocks per part
    return cut < 1 ? 1 : cut;
}
template <class Cfg>
inline void make_rows_plan(int64_t M, int64_t N, int64_t K, int sms, bool may_cut, RowsPlan* pl) {
    const int64_t NU = N / 8, P = sms < NU ? sms : NU, cut = rows_cut(N, K, sms, may_cut);
    int64_t runs;
    if (cut > 1) {
        runs = sms / cut;
        if (runs > NU) runs = NU;
    } else {
        runs = P * ((NU + 32 * P - 1) / (32 * P));   // none exceeds 256 rows
    }
    pl->cut = (int)cut;
    pl->T = (int)(runs * cut);
    pl->units = (int)(NU / runs);
    pl->more = (int)(NU % runs);
    const int rmax = (pl->units + (pl->more > 0)) * 8;
    pl->RB = rmax > 128 ? 2 : 1;
    pl->MN = (int)((M + 15) / 16) * 16;
    const int acols = (pl->RB * pl->MN + 31) & ~31;
    pl->S2 = (Cfg::kTmemCols - acols) / 64;
    if (pl->S2 > Cfg::kS2Max) pl->S2 = Cfg::kS2Max;
    pl->whalf = (rmax * (kRowCodeBytes + Cfg::kMeta) + 127) / 128 * 128;
    const int ks = 2 / pl->RB, x = ks * pl->MN * 128, slot = ks * pl->whalf, room = Cfg::kSmemBudget - Cfg::kFixed;
    while (pl->S2 > Cfg::G && room - pl->S2 * x < (pl->S2 + 2) * slot) --pl->S2;
    pl->S1 = (room - pl->S2 * x) / slot;
    if (pl->S1 > Cfg::kS1Max) pl->S1 = Cfg::kS1Max;
    pl->smem = Cfg::kFixed + pl->S2 * x + pl->S1 * slot;
}

// Up to sixteen tokens: CTAs of half an SM, so that the next launch's set up, fetch and expand beside this one's, where their main loop
// is short, since a CTA that has the SM to itself expands with half its warps.  Time of these over that of whole SMs, with quantization and
// alone, all of 1050 shapes but those that other kernels take:
//   more 128-channel tiles than half the SMs, K up to 1664 0.94, 0.73, to 2048 0.97, 0.80, to 3072 1.22, 0.88, to 6144 1.43, 0.93
//   K cut, k-blocks of a part: up to 8, M <= 12 0.98, 0.91; 13..16 1.08, 1.05
//                              9 or 10, M <= 4 1.00, 0.90; 5..12 1.05, 0.89
//                              11 to 14, M <= 4 1.03, 0.90 (11 of K up to 4352 0.95, 0.92, but see below); 5..12 1.14, 0.92
//                              more, M <= 4 1.22, 0.93; 5..12 1.26, 0.92
// us: (8, 4096, 4096) 7.6, 6.0 / 7.7, 7.6, (9, 4400, 3072) 7.2, 5.6 / 7.5, 7.5, (1, 5344, 3328) 7.3, 6.5 / 8.0, 7.4, (2, 13712, 1920) 6.7,
// 5.0 / 7.1, 6.6; (8, 6144, 4096), 11 k-blocks, 8.9, 7.3 / 8.5, 7.9, (8, 4096, 14336), 28, 16.2, 10.2 / 12.5, 11.9.
// Between launches that take whole SMs nothing starts beside these either.  Layers of 4096 channels, with a quantization per input, from a graph, all on whole SMs / so, us: q, k and v
// of 4096 and 1024 channels with 8 tokens 16.5 / 15.7; qkv, o, gate_up and down with 8 tokens, o here, 49.7 / 48.9 (called one by one 50.7 /
// 51.2), with q, k, v, gate and up apart 60.7 / 61.7; but qkv (11 k-blocks) here with 1 token 46.3 / 48.4, with 4 48.4 / 49.6.
// Hence not for a K of more than 6144, which down projections have, one layer per input: 2048 wide with 8192 between, 8 tokens, down here
// 26.5 / 28.1; nor more channels than half the SMs' tiles and K of 2048: the same block's gate_up here with 16 tokens 30.9 / 32.9.
inline bool half_rows_apply(int64_t M, int64_t N, int64_t K, int sms, bool may_cut) {
    if (M > 16) return false;
    if (2 * ((N + 127) / 128) > sms) return K <= 1664;
    const int64_t cut = rows_cut(N, K, sms, may_cut), blocks = (K / 128 + cut - 1) / cut;
    return cut > 1 && K <= 6144 && (M <= 4 ? blocks <= 10 : (M <= 12 && blocks <= 8));
}

enum DecodeKind {
    kDecodeNone,      // no number of SMs
    kDecodeDirect,    // linear_direct_kernel
    kDecodeWhole,     // whole tiles of the persistent kernel
    kDecodeCluster,   // persistent kernel, K cut between the CTAs of clusters
    kDecodeRows,      // linear_rows_kernel
    kDecodeRowsHalf   // ... CTAs of half an SM
};
struct DecodePlan {
    DirPlan direct;
    RowsPlan rows;
    int cluster;   // CTAs
};
template <int FMT>
inline DecodeKind decode_rows_choice(int64_t M, int64_t N, int64_t K, int sms, bool may_cut, DecodePlan* plan) {
    if (half_rows_apply(M, N, K, sms, may_cut)) {
        make_rows_plan<RowsSizes<FMT, true>>(M, N, K, sms, may_cut, &plan->rows);
        return kDecodeRowsHalf;
    }
    make_rows_plan<RowsSizes<FMT>>(M, N, K, sms, may_cut, &plan->rows);
    return kDecodeRows;
}
// 1..128 tokens on a prepacked layer.  `workspace`: the caller gave one that K can be cut through.  resident(size): clusters of
// that many CTAs that the device holds at once.
template <class Resident>
inline DecodeKind decode_choice(int64_t M, int64_t N, int64_t K, int fmt, int sms, bool workspace, bool y_on_host, Resident resident,
                                DecodePlan* plan) {
    if (sms <= 0) return kDecodeNone;
    // (linear_direct_kernel cuts K between the warps of a CTA.  Without a workspace K is never cut, which is how a
    // caller asks for the bits of a chain launch.  An output in host memory it writes in pieces of 32 bytes, which the
    // bus takes more slowly than rows: host to host, us, a kernel that writes rows / this, (4, 8192, 2048) 15.6 / 14.8, (8, 4096,
    // 3072) 17.1 / 16.8, (8, 6144, 2048) 15.9 / 17.2, (16, 6144, 2048) 19.1 / 24.1, (16, 8192, 1024) 19.3 / 24.0.)
    if (M <= 16 && workspace && (!y_on_host || M * N <= kHostFewOutputs) && direct_applies(M, N, K, fmt, sms, &plan->direct))
        return kDecodeDirect;
    if (whole_tiles_apply(M, N, K, fmt, sms, y_on_host)) return kDecodeWhole;
    if (M > 16) {
        // 17..128 tokens on a layer with few 128-row tiles and a long K: K cut between the CTAs of a cluster (cluster_kcut_pays;
        // us against the exchange through L2: (64, 2048, 4096) 6.9 / 12.9, (100, 512, 8192) 7.6 / 15.1), in the largest clusters
        // that are resident all at once: a second wave would cost more than the exchange through L2 saves.
        for (int cl = cluster_kcut_ctas(M, N, K, sms); cl >= 2 && cluster_kcut_pays(M, K, cl); --cl)
            if (resident(cl) >= (N + 127) / 128) {
                plan->cluster = cl;
                return kDecodeCluster;
            }
        // (With zero-points whole tiles are the better ones where clusters do not pay, us against rows: (120, 2048, 2944) 9.6 / 10.9, (54,
        // 6336, 2304) 7.5 / 8.3, (126, 7776, 4864) 14.6 / 15.0; sign-magnitude level, (98, 3488, 2688) 9.0 / 9.0.)
        if (fmt == kFmtTiled && 2 * ((N + 127) / 128) <= sms && K <= 5120) return kDecodeWhole;
    }
    const bool may_cut = M <= 16 && workspace;
    return fmt == kFmtTiledSignMag ? decode_rows_choice<kFmtTiledSignMag>(M, N, K, sms, may_cut, plan)
                                   : decode_rows_choice<kFmtTiled>(M, N, K, sms, may_cut, plan);
}

}  // namespace w4a8
