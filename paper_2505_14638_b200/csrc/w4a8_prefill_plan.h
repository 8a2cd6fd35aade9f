// Plans of the prepacked layers that are chosen by cost models, and the order in which CTA pairs take their tiles: host code
// without CUDA, but for the tile order, which the kernel uses as well.
#pragma once

#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define W4A8_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define W4A8_HOST_DEVICE inline
#endif

namespace w4a8 {

constexpr int kMaxSMs = 160;  // upper bound used to size workspaces without touching a device

// Layout of every w4a8_linear workspace, whatever kernel and shape use it: a control area of fixed
// size at the start (tile counters of the persistent kernel; K-cut counters and placement state
// of the split-N kernel), which every launch leaves zero-filled, and behind it the data (partial
// sums), which may be left in any state.  With the control area at a shape-dependent size, one
// call's left-over partial sums could sit where the next call -- another layer, another kernel
// -- expects zeroed counters; callers do share one workspace between the layers of a model.
constexpr size_t kLinearCtlBytes = 65536;
// The split-N kernel's 2 KB (K-cut counters, placement state -- whose generation word stays non-zero
// by design) sit at the END of the control area, the persistent kernel's tile counters at its start.
constexpr size_t kLinearCtlSplitN = kLinearCtlBytes - 2048;

struct SkPlan {
    int bnx, TM, TN;
    int aligned;   // 1: whole tiles per CTA, nothing shared; 0: equal slices of the (tile, k-block) space
    int64_t P;     // CTAs
    int64_t U;
    size_t counter_bytes, workspace_bytes;
};

// Tile t of a CTA pair's schedule -> channel tile and token tile.  Token tiles are taken in bands of kPairBand: the tiles in
// flight at a time then cover a few token tiles and a few channel tiles, and what they read fits L2 (with token tiles running
// through (8192, 28672, 8192) reads all 67 MB of X8 again for every four channel tiles).  A last token tile that takes half as
// long as the others (256 x 512 tiles, at most 256 tokens in it) is a band of its own: `full` token tiles come first, so that
// the last round of tiles holds short ones where it can.  (1152, 7648, 2560) 32.9 -> 27.3 us, (526, 14128, 2560) 33.0 -> 27.3.
// (`full` is the host's: worked out in the kernel, the same loops took 3 % longer, (2048, 4096, 4096) 41.2 -> 42.2 us.)
constexpr int kPairBand = 8;
W4A8_HOST_DEVICE int pair_full_tiles(int64_t M, int tokens, int TM) { return tokens > 256 && M - (int64_t)(TM - 1) * tokens <= 256 ? TM - 1 : TM; }
W4A8_HOST_DEVICE void pair_tile(int t, int full, int TN, int& nt, int& mt) {
    const int per = kPairBand * TN, band = t / per;
    int first = band * kPairBand, u = t - band * per;
    int width = full - first < kPairBand ? full - first : kPairBand;
    if (t >= full * TN) {
        first = full;
        u = t - full * TN;
        width = 1;
    }
    nt = u / width;
    mt = first + (u - nt * width);
}

// Time of 256 x 512 tiles on `pairs` pairs, in half rounds: pair c takes tiles c, c + pairs, ..., and one of at most 256 tokens
// takes half as long.
inline int64_t pair_half_rounds(int64_t M, int64_t N, int64_t pairs) {
    const int64_t TN = (N + 255) / 256, TM = (M + 511) / 512, tiles = TN * TM, rounds = (tiles + pairs - 1) / pairs;
    const int64_t full = TN * pair_full_tiles(M, 512, (int)TM);   // pair 0 has most of them, and a tile of each round
    return rounds + (full + pairs - 1) / pairs;
}

// Token-tile width and schedule of the persistent kernel on prepacked weights from a cost model, in microseconds; returns
// the time.  Whole tiles per CTA cost rounds x (k-blocks x step + drain); where there are fewer tiles than half the CTAs and
// a number of CTAs per tile divides the k-blocks, that many CTAs share a tile and exchange partial sums, which costs about
// as much as 30 k-blocks.  Fitted, with the constants of the CTA pairs (see prefill_choice), to 656 + 410 measured (M, N,
// K) of all alternatives: the alternative chosen takes 0.5 % longer than the fastest on average, 9 % at most from K = 1024
// on.  Equal slices of the (tile, k-block) space and tiles of 256 tokens, which earlier versions had, are nowhere the
// fastest by more than 4 %.
inline double make_sk_plan(int64_t M, int64_t N, int64_t K, int sms, SkPlan* pl) {
    const int64_t KB = K / 128;
    const int64_t TN = (N + 127) / 128;
    const int64_t cap = sms < kMaxSMs ? sms : kMaxSMs;
    double best = 1e30;
    for (int bnx = 128; bnx >= 64; bnx >>= 1) {
        if (bnx > 64 && bnx / 2 >= M) continue;  // more than half of the tile would be padding
        const int64_t TM = (M + bnx - 1) / bnx, Tt = TM * TN;
        const double step = bnx == 64 ? 0.207 : 0.247, drain = bnx == 64 ? 0.46 : 0.89;
        double t = (double)((Tt + cap - 1) / cap) * ((double)KB * step + drain) + 1.8;
        int64_t P = cap < Tt ? cap : Tt;
        bool whole = true;
        const int64_t per = cap / Tt;   // CTAs per tile
        // (tile counters must fit the control area)
        if (per >= 2 && KB % per == 0 && 2 * (size_t)Tt * sizeof(unsigned int) <= kLinearCtlSplitN) {
            const double t_k = (double)(KB / per) * step + 7.7;
            if (t_k < t) {
                t = t_k;
                P = Tt * per;
                whole = false;
            }
        }
        if (t < best) {
            best = t;
            pl->bnx = bnx;
            pl->TM = (int)TM;
            pl->TN = (int)TN;
            pl->U = Tt * KB;
            pl->aligned = whole ? 1 : 0;
            pl->P = P;
        }
    }
    // arrivals and finished reducers per tile live in the control area; the size asked of the caller
    // covers every tile width and any SM count up to kMaxSMs, so that the query needs no device
    pl->counter_bytes = kLinearCtlBytes;
    pl->workspace_bytes = kLinearCtlBytes + (size_t)kMaxSMs * 2 * 256 * 128 * sizeof(float);
    return best;
}

// CTA pairs against the persistent kernel for a problem of more than 128 tokens: 0 = persistent kernel (its plan in `pl`),
// 1 = tiles of 256 channels x 256 tokens, 2 = 256 x 512, 3 = 256 x 256 with K cut between the two pairs of a cluster of four
// CTAs.  Times in microseconds, from the same fit as make_sk_plan's: a k-block of a 256 x 256 tile takes a pair 0.244, of a
// 256 x 512 tile 0.489 (a round that holds only tiles of at most 256 tokens half of that); drain per tile, launch and fill
// per call.  Measured, us, sign-magnitude weights not in L2 (before / now, the choice in brackets): (8192, 28672, 8192) 2011 /
// 1500 [2], (2048, 4096, 4096) 36.3 / 34.7 [2], (1531, 28672, 4096) 208 / 171 [2], (1531, 4096, 14336) 121 / 95 [2], (1024,
// 28672, 4096) 152 / 121 [2], (512, 6144, 4096) 18.4 / 15.9 [1], (512, 28672, 4096) 71 / 63 [2], (512, 4096, 14336) 45.2 / 33.0
// [3], (256, 4096, 4096) 16.5 / 10.9 [3]; (512, 4096, 4096) 12.2 / - / 14.1 on pairs [0].
inline int prefill_choice(int64_t M, int64_t N, int64_t K, int sms, int quads, SkPlan* pl) {
    const int64_t KB = K / 128, pairs = sms / 2, TN = (N + 255) / 256;
    double best = make_sk_plan(M, N, K, sms, pl);
    int choice = 0;
    const int64_t t1 = TN * ((M + 255) / 256);
    const int64_t rounds1 = (t1 + pairs - 1) / pairs;
    double t = (double)rounds1 * ((double)KB * 0.244 + 2.1) + 3.1;
    // (back to back, at the power cap, where all pairs work throughout: it expands twice the weights)
    if (rounds1 >= 2) t *= 1.1;
    if (t < best) {
        best = t;
        choice = 1;
    }
    t = 0.5 * (double)pair_half_rounds(M, N, pairs) * ((double)KB * 0.489 + 2.3) + 6.8;
    if (t < best) {
        best = t;
        choice = 2;
    }
    if (t1 <= quads && KB >= 8) {   // (a second round of them would cost more than the cut saves)
        t = (double)((KB + 1) / 2) * 0.244 + 7.3;
        if (t < best) choice = 3;
    }
    return choice;
}

}  // namespace w4a8
