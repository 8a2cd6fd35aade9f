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
}  // namespace w4a8
