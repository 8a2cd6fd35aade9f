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
// size at the start (tile counters of the persistent kernel; K-cut counters of
// linear_rows_kernel), which every launch leaves zero-filled, and behind it the data (partial
// sums), which may be left in any state.  With the control area at a shape-dependent size, one
// call's left-over partial sums could sit where the next call -- another layer, another kernel
// -- expects zeroed counters; callers do share one workspace between the layers of a model.
constexpr size_t kLinearCtlBytes = 65536;
// The K-cut counters of linear_rows_kernel sit in the last 2 KB of the control area, the persistent kernel's tile counters at
// its start.
constexpr size_t kLinearCtlRows = kLinearCtlBytes - 2048;

// What w4a8_linear_workspace_bytes asks for and w4a8_linear requires for more than 128 tokens on prepacked weights, whatever
// arrangement runs (most use none of it): a bound on what the persistent kernel ever used, for any SM count up to kMaxSMs.  It
// does not follow the plans, so that a workspace that was accepted stays accepted and one that was refused stays refused.
constexpr size_t kSkWorkspaceBytes = kLinearCtlBytes + (size_t)kMaxSMs * 2 * 256 * 128 * sizeof(float);

struct SkPlan {
    int bnx, TM, TN;
    int per;       // CTAs per tile (1: whole tiles, a run of them per CTA)
    int64_t P;     // CTAs
    size_t counter_bytes;
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

// Tiles of 256 x 512 that the busiest of `pairs` pairs works on (pair c takes tiles c, c + pairs, ...): those with two
// accumulators, or those with one.
inline int64_t pair_rounds(int64_t M, int64_t N, int64_t pairs, bool two) {
    const int64_t TN = (N + 255) / 256, TM = (M + 511) / 512, full = TN * pair_full_tiles(M, 512, (int)TM);
    const int64_t of_two = (full + pairs - 1) / pairs;
    return two ? of_two : (TN * TM + pairs - 1) / pairs - of_two;
}

// More than 128 tokens on prepacked weights: the arrangements there are.
enum PrefillKind {
    kPairs256,     // CTA pairs, tiles of 256 channels x 256 tokens
    kPairs512,     // 256 x 512
    kPairsKCut,    // 256 x 256 with K cut between the two pairs of a cluster of four CTAs
    kWhole64,      // persistent kernel, whole tiles of 128 channels x 64 tokens per CTA
    kWhole128,     // x 128
    kWhole256,     // x 256
    kCut128,       // persistent kernel, several CTAs per tile of 128 x 128, which exchange partial sums through the workspace
    kCut256,       // 128 x 256
    kPrefillKinds
};

// Time of a launch in microseconds, with the activation quantization before it:
//   rounds of tiles x max(k-blocks x step + drain, least) + fixed + full x (share of the SMs that the first round takes)^4
// `least`: the drain of a tile that its k-blocks do not cover (kPairs512: the time of a tile with one accumulator as a part of
// one with two).  `full`: a launch that leaves SMs free lets the next one set up beside it, which is why 69 CTAs with 128 tokens
// each take less time than 138 with 64, (383, 2896, 1536) 7.7 against 8.3 us.
struct PlanCost {
    double step, drain, fixed, full, least;
};
// Sign-magnitude and generic format.  (The latter's were fitted when its expansion took twice the instructions it takes now.  Timed
// again with every arrangement, 200 shapes, each 30 ms warm, they choose 2.5 % above the fastest of the eight on average, 1.18 times at
// worst, where two timings of one arrangement lie up to 14 % apart.)
constexpr PlanCost kPlanCost[2][kPrefillKinds] = {
    {
        {0.373, 3.16, 2.71, 0.19, 0.00},    // pairs, 256 x 256
        {0.887, 3.28, 4.52, -0.91, 0.52},   // pairs, 256 x 512
        {0.309, 0.00, 8.83, 6.79, 0.00},    // pairs, 256 x 256, K cut
        {0.276, 0.22, 2.48, 2.31, 1.44},    // whole tiles, 128 x 64
        {0.300, 0.81, 2.85, 1.78, 2.12},    // whole tiles, 128 x 128
        {0.524, 2.18, 3.35, 0.09, 0.25},    // whole tiles, 128 x 256
        {0.356, 0.00, 11.48, 0.02, 0.00},   // K cut, 128 x 128
        {0.546, 0.00, 14.63, 0.04, 0.00},   // K cut, 128 x 256
    },
    {
        {0.486, 2.31, 2.68, 0.38, 0.00},    // pairs, 256 x 256
        {0.809, 3.66, 3.82, -0.14, 0.60},   // pairs, 256 x 512
        {0.447, 0.00, 7.98, 4.67, 0.00},    // pairs, 256 x 256, K cut
        {0.356, 0.38, 2.56, 2.75, 1.24},    // whole tiles, 128 x 64
        {0.376, 1.06, 2.42, 2.31, 2.52},    // whole tiles, 128 x 128
        {0.539, 1.77, 3.99, 1.72, 0.09},    // whole tiles, 128 x 256
        {0.467, 0.00, 9.15, 2.85, 0.00},    // K cut, 128 x 128
        {0.643, 0.00, 7.44, 9.09, 0.00},    // K cut, 128 x 256
    },
};

inline double plan_time(const PlanCost& c, double rounds, int64_t steps, double taken) {
    const double tile = (double)steps * c.step + c.drain, share = taken < 1.0 ? taken : 1.0;
    return rounds * (tile > c.least ? tile : c.least) + c.fixed + c.full * share * share * share * share;
}

// The arrangement with the least time by that model; `pl`: the persistent kernel's plan where it is one of those.  `quads`:
// clusters of four CTAs that the device holds at once (a second round of them costs more than the cut saves).
// The constants are fitted to 1778 (M, N, K) in both formats, M 129 to 8192, N 1024 to 28672, K 1024 to 14336 and some shorter
// ones: every arrangement in turn for a few milliseconds, quantization and linear layer back to back, weights not in L2; and
// to 190 of them run for a quarter of a second each, at the power cap.  The arrangement taken is 0.5 % slower than the fastest
// on average, 15 % at most; it is slower than the kernels before CTA pairs by more than 3 % at 24 of the 3542, by 11 % at most
// ((635, 1216, 2944) generic 11.8 -> 13.3 us), and 1.17 times as fast on average.
// The model before this one had the same constants for both formats, took 36 clusters of four for granted and lacked 256-token
// tiles and uneven cuts of K: (241, 8592, 5248) 28.6 -> 17.5 us, (1488, 1376, 10496) 47.0 -> 31.0, (151, 1072, 12416) 22.1 -> 15.5,
// (1196, 3680, 4864) generic 33.5 -> 28.3, (1531, 4096, 14336) 104.8 -> 97.2.
inline PrefillKind prefill_choice(int64_t M, int64_t N, int64_t K, bool signmag, int sms, int quads, SkPlan* pl) {
    const PlanCost* cost = kPlanCost[signmag ? 0 : 1];
    const int64_t KB = K / 128, cap = sms < kMaxSMs ? sms : kMaxSMs, pairs = sms / 2;
    PrefillKind kind = kPrefillKinds;
    double best = 1e30;
    auto better = [&](PrefillKind k, double t) {
        if (t >= best) return false;
        best = t;
        kind = k;
        return true;
    };
    const int64_t TNp = (N + 255) / 256, t1 = TNp * ((M + 255) / 256), TM2 = (M + 511) / 512;
    const int64_t rounds1 = (t1 + pairs - 1) / pairs, full = TNp * pair_full_tiles(M, 512, (int)TM2);
    // Sign-magnitude launches of some 35 us and more, one after the other, run at the power cap, where expanding the weights twice
    // as often as 256 x 512 tiles with two accumulators do costs clock: a quarter of a second of (2048, 4096, 4096) 39.4 against
    // 38.6 us, of (1531, 28672, 4096) 178 / 170, of (8192, 28672, 8192) 1669 / 1632.
    double capped = 0.0;
    if (signmag) capped = rounds1 >= 8 ? 0.18 : ((double)M * (double)N * (double)K >= 3e10 ? 0.09 : 0.0);
    capped = 1.0 + capped * (double)full / (double)(TNp * TM2);
    better(kPairs256, plan_time(cost[kPairs256], (double)rounds1, KB, (double)t1 / (double)pairs) * capped);
    {
        // (`least` of this arrangement is a factor, see PlanCost)
        PlanCost c = cost[kPairs512];
        const double rounds = (double)pair_rounds(M, N, pairs, true) + c.least * (double)pair_rounds(M, N, pairs, false);
        c.least = 0.0;
        better(kPairs512, plan_time(c, rounds, KB, (double)(TNp * TM2) / (double)pairs));
    }
    if (t1 <= quads && KB >= 8) better(kPairsKCut, plan_time(cost[kPairsKCut], 1.0, (KB + 1) / 2, 2.0 * (double)t1 / (double)pairs));
    for (int i = 0; i < 3; ++i) {
        const int bnx = 64 << i;
        if (bnx > 64 && bnx / 2 >= M) continue;  // more than half of the tile would be padding
        const int64_t TM = (M + bnx - 1) / bnx, TN = (N + 127) / 128, tiles = TM * TN, per = cap / tiles;
        int64_t ctas = 0;   // per tile
        if (better((PrefillKind)(kWhole64 + i), plan_time(cost[kWhole64 + i], (double)((tiles + cap - 1) / cap), KB, (double)tiles / (double)cap))) ctas = 1;
        if (i > 0 && per >= 2 && KB >= 2 * per &&
            better((PrefillKind)(kCut128 + i - 1), plan_time(cost[kCut128 + i - 1], 1.0, (KB + per - 1) / per, (double)(tiles * per) / (double)cap)))
            ctas = per;
        if (ctas == 0) continue;
        pl->bnx = bnx;
        pl->TM = (int)TM;
        pl->TN = (int)TN;
        pl->per = (int)ctas;
        pl->P = ctas == 1 ? (tiles < cap ? tiles : cap) : tiles * ctas;
        pl->counter_bytes = ctas == 1 ? 0 : kLinearCtlBytes;
    }
    return kind;
}

}  // namespace w4a8
