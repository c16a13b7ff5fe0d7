// How a consumer call is spread over the GPU, and the scratch that takes (host only).
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "tree_layout.h"

namespace wdf {

// Most scratch of a call's node values or parts' sums; the context's pool keeps as much
// between calls.
constexpr int64_t kScratchBytes = 320ll << 20;

struct ExplainPlan {
    int splits;             // 0: node values (k_values, k_sum_values), else the tile kernel with its tiles'
                            // parts on that many blocks
    int64_t rows;           // rows of a launch: with several splits as many as the scratch holds
    size_t scratch_floats;  // node values, or with several splits the parts' sums of a launch
};

// The plan of n rows against T trees of depth D, tiles of tile_rows rows, per_sm of them on
// each of sms SMs at a time.  The least of estimated microseconds:
//  - tile kernel: its waves of resident blocks times a tile's walk of its trees, 0.034 us per
//    tree and leaf position at full occupancy, down to half of it with a block to itself;
//    split, the parts' sums are written and read once more;
//  - node values: 1.4 ps (depth 8: 2.2) per row and flush position, 8 ps per row and feature.
// Measured (node values / parts on blocks / one block a tile): 200 trees of depth 6, 127 features,
// 1,000 rows 29 / 68 / 211 us, 2,000 rows 47 / 68, 4,000 rows 88 / 82, 8,000 rows - / 118 / 224; 1000
// trees of depth 8, 100 rows 99 / 706; 500 trees of depth 7, 777 rows 88 / 156 / 1149; 50 trees of
// depth 4, 255 features, 20,000 rows 82 / 51.  The line is drawn a little early for calls of about
// 4,000 rows of shallow trees (500 of depth 4: 60 / 79) and 1,000 of 100 trees of depth 8 (74 / 92).
// Neither form takes more than kScratchBytes: node values are not chosen beyond, and split tiles
// run one slice of the rows after another (a multiple of 128 rows).  293,300 rows, 1000 trees of
// depth 8 and 134 features: 63.8 ms with the parts of all rows at once (1.26 GB), 64.5 in slices,
// 67.5 with whole tiles; 100,000 rows, 400 trees of depth 8 and 500 features 22.3 (1.6 GB), 22.8
// and 27.9 (blocks at work on the same part share its folded vectors in the L2 cache).
// values: a row block's codes fit the shared memory of the node values' kernel.
inline ExplainPlan explain_plan(int D, int64_t n, int T, int F, int tile_rows, int sms, int64_t per_sm,
                                bool values = true) {
    const int P = explain_parts(T, D);
    const int64_t room = (int64_t)sms * per_sm;
    const double walk = 0.034 * T * (1 << D);
    ExplainPlan best{1, n, 0};
    double least = 0.0;
    for (int s = 1; s <= P; ++s) {
        int64_t rows = n;
        if (s > 1) {  // equal slices
            const int64_t most = kScratchBytes / 4 / ((int64_t)P * F) / 128 * 128;
            if (most == 0) break;
            const int64_t slices = (n + most - 1) / most;
            if (slices > 1) rows = ((n + slices - 1) / slices + 127) / 128 * 128;
        }
        double cost = s > 1 ? 2e-6 * (double)P * (double)n * F : 0.0;
        for (int64_t r0 = 0; r0 < n; r0 += rows) {
            const int64_t items = (std::min(rows, n - r0) + tile_rows - 1) / tile_rows * s;
            const double full = (double)items / (double)room;
            const double waves = (double)((items + room - 1) / room) * ((P + s - 1) / s) / P;
            cost += waves * walk * (full < 1.0 ? 0.5 + 0.5 * full : 1.0) + (s > 1 ? 4.0 : 0.0);
        }
        cost += 15.0;
        if (s == 1 || cost < least) {
            best = ExplainPlan{s, rows, s > 1 ? (size_t)P * (size_t)rows * (size_t)F : 0};
            least = cost;
        }
    }
    const int64_t rows = (n + 31) / 32 * 32, positions = (int64_t)T * flush_len(D);
    if (values && rows <= kScratchBytes / 4 / positions) {
        const double cost = 20.0 + (double)rows * ((D == 8 ? 2.2e-6 : 1.4e-6) * (double)positions + 8e-6 * F);
        if (cost < least) best = ExplainPlan{0, n, (size_t)(rows * positions)};
    }
    return best;
}

// Bytes of a call's scratch: its rows' codes, then the plan's floats (from scratch_at on).
inline size_t scratch_at(size_t code_bytes) { return (code_bytes + 255) & ~(size_t)255; }

// Takes the scratch of a call by alloc(bytes).  Where it does not fit (alloc returns no_memory)
// the call runs with whole tiles, which need only the codes.
template <class Error, class Alloc>
Error take_scratch(ExplainPlan *plan, int64_t n, size_t code_bytes, Error no_memory, Alloc alloc) {
    Error e = alloc(scratch_at(code_bytes) + plan->scratch_floats * sizeof(float));
    if (e == no_memory && plan->scratch_floats > 0) {
        *plan = ExplainPlan{1, n, 0};
        e = alloc(scratch_at(code_bytes));
    }
    return e;
}

}  // namespace wdf
