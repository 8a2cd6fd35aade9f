// The order in which dpq_kernel takes its tasks: host and device code, which a host test compiles as well.
#pragma once

#ifdef __CUDACC__
#define W4A8_HOST_DEVICE __host__ __device__
#else
#define W4A8_HOST_DEVICE
#endif

namespace w4a8 {

// The order of the tasks.  Step b: block b, then applications of errors that earlier blocks left.  Blocks come in panels of D = 8, 4, 2
// or 1, by the rounds of CTAs that a step's tiles make, whose errors go to the columns behind the panel together (a tile's weights
// are read and written, and a task started, once per 128 D values of q): `far`, in parts, one in each step of the next panel, that
// panel's own columns first.  (Panels of at most two / four / eight blocks, us: (4096, 14336) 17830 / 16990 / 16870, (8192, 8192)
// 12550 / 12010 / 11890; four and two blocks from 8 and 4 rounds on instead of 4 and 2: 17350, 12185.)  Inside a
// panel a block's errors go to the columns up to the first one behind it (`near`), one block at a time.  The block's own task adds
// the errors of the block before.  Every column sees the errors in ascending order.
struct DpqTrail {
    int errors;   // first block whose errors are applied
    int blocks;   // how many
    int first;    // first column block
    int count;    // column blocks
};
struct DpqSteps {
    int G, row_tiles, slots;
    int b;                    // step (-1: before the first)
    int D, panel, end;        // blocks panel .. end - 1 = panel + D - 1
    int left;                 // column blocks, the last ones, that the errors of the panel before have still to be applied to
    DpqTrail far, near;
    W4A8_HOST_DEVICE void next() {
        ++b;
        const int n = G - 1 - b;   // column blocks behind block b
        if (b == end) {
            const long long tiles = (long long)row_tiles * n;
            const long long rounds = tiles / slots;
            const int before = D, want = rounds >= 6 ? 8 : (rounds >= 4 ? 4 : (rounds >= 2 ? 2 : 1));
            D = b == 0 || want < before ? want : before;
            panel = b;
            end = b + D;
            far = {b - before, before, 0, 0};
            left = b > 0 ? n : 0;
        }
        const int j = b - panel, part = (left + D - j - 1) / (D - j);
        far.first = G - left;
        far.count = j == 0 && part < D ? (left < D ? left : D) : part;
        left -= far.count;
        near = {b - 1, 1, b + 1, j == 0 ? 0 : (n < D - j ? n : D - j)};
    }
};
// How the n tiles of a Hessian (the upper triangle of nb x nb) are dealt out: `whole` tiles are taken by a CTA each; of the others, all
// off the diagonal, a CTA takes the first `cut` tokens of `bundle` tiles, and in a second launch the other tokens of one.  The first
// launch hands its sums over in the place of the tile's mirror image, which has to be all there (K % 128 == 0).  An entry stays one
// chain over the tokens in order.
// Two CTAs to an SM share its FMA pipes, and one alone has nearly all of them, so that the time in tiles per SM is ceil(n / sms) where
// all tiles are whole, 4 for 528 tiles on 148 SMs, which 3.57 would do.  With bundles of k tiles, each a k-th of its tokens, a bundle
// takes as long as a tile, and the second launch (k - 1) / k of that for each CTA that an SM has of it.  The least of these is taken
// where it spares 1.5 % of the time (the loop over a bundle's tiles), a twelfth of a tile and what 110 tokens of a tile take (10 us: the
// sums go out and come back): (256, 4480) 138.8 whole, 140.7 shared, (823, 4736) 372 and 375.  Measured, us per call, whole / shared: (T, K) = (1024, 3072) 282 / 238, (1024, 3584) 282 / 274,
// (640, 4096) 240 / 230, (1024, 4096) 368 / 353, (2048, 4096) 711 / 670, (1024, 4480) 458 / 422, (2048, 5120) 1059 / 1027, (1024, 8192)
// 1329 / 1309.
struct HessianSplit {
    int whole, bundle, cut;
};
inline HessianSplit hessian_split(long long nb, long long sms, long long tokens, int chunk) {
    const long long n = nb * (nb + 1) / 2, chunks = tokens / chunk;
    HessianSplit s = {(int)n, 0, 0};
    if (sms <= 0) return s;
    const double whole = (double)((n + sms - 1) / sms);
    double best = 0.985 * whole - 0.08 - 110.0 / (double)tokens;
    for (int k = 2; k <= 8 && chunks >= 8 * k; ++k)
        for (int rounds = 1; rounds <= 2; ++rounds) {
            const long long split = rounds * sms < n - nb ? rounds * sms : n - nb;
            const double time = (double)((n - split + (split + k - 1) / k + sms - 1) / sms) + rounds * (k - 1.0) / k;
            if (time >= best) continue;
            best = time;
            s.whole = (int)(n - split);
            s.bundle = k;
            s.cut = (int)(chunks / k * chunk);
        }
    return s;
}

}  // namespace w4a8
