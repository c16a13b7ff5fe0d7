// Per-tree records shared by the host packer and the kernels (plain structs, no device
// code), and the order in which the consumer kernel adds a tree's node values into phi.
//
// Decision codes.  Every real inner node tests x[f] < thr (Def. "decision_tree").  The
// packer sorts the distinct thresholds of each feature and cuts the sorted list into
// "code columns" of at most 2^kSliceBits - 1 thresholds.  A row's code in column c is the
// number of the column's thresholds u with u <= x (the column's threshold count when x is
// NaN).  A node whose threshold is the k-th of its column (rank k, 0-based) sends the row
// left exactly when code <= k, because the thresholds are sorted: x < u_k  <=>  fewer than
// k + 1 of them are <= x.  A NaN threshold never sends a row left (rank -1).  The kernels
// stage codes instead of floats: half a byte to one and a half bytes per column and row
// instead of four bytes per feature.
//
// Flush sequence of a tree of depth D, the order in which the consumer kernel adds node
// values into phi.  The bottom subtrees come in groups of GS = gather_group(D) consecutive
// ones, those of one unit (below); NG groups.  Per group: the three inner nodes r, 2r+1, 2r+2
// of its subtrees, two subtrees to a batch of eight positions (a pair whose nodes are all
// pass-through nodes, as below an early leaf, is skipped as a whole), then the GS - 1 inner
// nodes above them inside the group (heap order within it), padded to a batch.  After the
// groups: the NG - 1 nodes above them, padded to a batch.  Batch b is positions [8b, 8b + 8).
// A batch whose real features are all distinct can read all its phi values before writing
// any.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define WDF_HD __host__ __device__
#else
#define WDF_HD
#endif

namespace wdf {

// Sliced codes.  The codes are stored bit by bit: the rows of a 32-row block give one 32-bit word per code bit (bit r of the word = row r), four words
// (a "quad", 16 bytes) per four code bits, and a node's decision for all 32 rows is
//   le = all ones; for every code bit from the least significant: le = majority(~bit, rank bit, le)
// (code <= rank), eight three-input logic instructions for 32 decisions.  Columns are sorted
// by their number of code bits, largest first, and padded to packs of eight columns of equal
// width; quad k of column c lies at quad index qbase[k] + c of the block, so columns with
// more than k quads are exactly the first ones.  A column takes at most kSliceBits bits;
// a feature with more thresholds is cut into several columns.
//
// The 31 inner nodes of a height-5 subtree, one per lane of a warp, are a "unit": a tree of
// depth D >= 5 has 2^(D-5) of them, side by side below its 2^(D-5) - 1 top nodes; a smaller
// tree is one unit of 2^D - 1 nodes.  Lanes of a unit with S bottom subtrees: the S - 1 nodes
// above them in heap order, then per subtree its root's left child, right child and the root,
// so that the three low bits of a row's entry lie side by side in its decision word.  Lane 31
// of unit u carries top node u.
constexpr int kSliceBits = 12;
constexpr int kSliceGroupPacks = 16;      // most packs (of eight columns) encoded together
constexpr int kSliceGroupFloats = 16384;  // most thresholds of an encoding group (one pack may exceed it)

// A lane's node of a unit: its column and the rank it compares with.
struct UnitNode {
    uint32_t at;    // unit_at: column index | quads << 24 (0: none to read) | start << 28 (the comparison's start:
                    // 1 when a code equal to the rank goes left; without quads it is the decision itself)
    uint32_t rank;  // bit 7 - k of byte b is bit 4k + b of the rank
};
// Columns that a node can name; an ensemble with more of them cannot be counted or explained.
constexpr int64_t kMostColumns = (int64_t)1 << 24;
WDF_HD constexpr uint32_t unit_at(uint32_t column, uint32_t quads, uint32_t start) {
    return column | quads << 24 | start << 28;
}
WDF_HD constexpr int unit_column(uint32_t at) { return (int)(at & (uint32_t)(kMostColumns - 1)); }
WDF_HD constexpr int unit_quads(uint32_t at) { return (int)((at >> 24) & 15u); }
WDF_HD constexpr uint32_t unit_start(uint32_t at) { return (at >> 28) & 1u; }
// One column of a pack: its feature and its number of thresholds (the code of a NaN).
struct SliceCol {
    int32_t feature, count;
};
// Eight columns: their thresholds are search trees of 2^levels - 1 nodes (root at 1, children
// of i at 2i and 2i + 1, NaN after the column's thresholds) at sthr[first + (j << levels)].
struct SlicePack {
    int32_t first, levels;
};
// Packs [pack0, pack1) whose thresholds [thr0, thr0 + thr_n) one encoding block keeps in
// shared memory.
struct SliceGroup {
    int32_t pack0, pack1, thr0, thr_n;
};
WDF_HD constexpr int unit_height(int D) { return D < 5 ? D : 5; }
WDF_HD constexpr int unit_top(int D) { return D > 5 ? D - 5 : 0; }      // levels above the units
WDF_HD constexpr int units_per_tree(int D) { return 1 << unit_top(D); }
WDF_HD constexpr int unit_subtrees(int D) { return 1 << (unit_height(D) - 2); }
// Heap index of the node of lane i of unit u (i < 2^unit_height - 1).
WDF_HD inline int unit_node(int D, int u, int i) {
    const int S = unit_subtrees(D), top = unit_top(D);
    if (i < S - 1) {
        int l = 0;
        while ((2 << l) <= i + 1) ++l;
        return (1 << (top + l)) - 1 + (u << l) + (i - ((1 << l) - 1));
    }
    const int r = (1 << (D - 2)) - 1 + u * S + (i - (S - 1)) / 3, c = (i - (S - 1)) % 3;
    return c == 2 ? r : 2 * r + 1 + c;
}

// One real inner node of a tree, in heap order (the interaction kernels).
struct NodeRec {
    int32_t col;      // the node's code column
    int32_t rank;     // left when code <= rank; -1 for a NaN threshold
    // the node's decision bit: trees of at most 64 inner nodes (depth <= 6) carry it in
    // two words (bit_lo: heap index < 32, bit_hi: the rest), deeper trees as the bit
    // within its word (bit_lo, bit_hi = 0)
    uint32_t bit_lo, bit_hi;
};

struct TreeMeta {
    uint32_t pt[8];   // bit v of word v/32: inner node v is a pass-through node (always left)
    uint64_t live;    // bit s: bottom subtree s has a non-zero leaf
    uint64_t flush;   // bit b: consumer flush batch b repeats no real feature
    uint8_t wend[8];  // NodeRec index one past the last node of word w
    uint64_t real;    // bit b: consumer flush batch b holds a real (not pass-through) node
};
static_assert(sizeof(NodeRec) == 16, "NodeRec is one 16-byte load");
static_assert(sizeof(TreeMeta) == 64, "TreeMeta layout");

// Slots per entry of the folded slot vectors: D - 2 ancestors and the three nodes of the
// bottom subtree.  An entry is one 16- or 32-byte vector of slots; at depth 8, whose nine
// slots do not fit, the root's slot is kept apart (one float per entry after all vectors).
WDF_HD constexpr int slots_per_entry(int D) { return (D + 1) <= 4 ? 4 : 8; }
WDF_HD constexpr int extra_slots(int D) { return D == 8 ? 1 : 0; }
// Bottom subtrees per gather group: those of a unit, whose slot vectors are in flight together
// in at most 64 registers.
WDF_HD constexpr int gather_group(int D) { return 1 << (unit_height(D) - 2); }
WDF_HD constexpr int pad8(int n) { return (n + 7) & ~7; }
WDF_HD constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }
WDF_HD constexpr int flush_groups(int D) { return (1 << (D - 2)) / gather_group(D); }
WDF_HD constexpr int flush_group_bottom(int D) { return 8 * ((gather_group(D) + 1) / 2); }
WDF_HD constexpr int flush_group_len(int D) { return flush_group_bottom(D) + pad8(gather_group(D) - 1); }
WDF_HD constexpr int flush_len(int D) { return flush_groups(D) * flush_group_len(D) + pad8(flush_groups(D) - 1); }
WDF_HD constexpr int flush_batches(int D) { return flush_len(D) / 8; }

// Heap index of the node at flush position i, -1 for padding.
WDF_HD inline int flush_node(int D, int i) {
    const int NS = 1 << (D - 2), GS = gather_group(D), NG = NS / GS, GL = flush_group_len(D);
    if (i >= NG * GL) {
        const int u = i - NG * GL;
        return u < NG - 1 ? u : -1;
    }
    const int g = i / GL, k = i - g * GL;
    if (k < flush_group_bottom(D)) {
        const int s = 2 * (k / 8) + k % 8 / 3, c = k % 8 % 3;  // two subtrees to a batch
        if (k % 8 >= 6 || s >= GS) return -1;
        const int r = NS - 1 + g * GS + s;
        return c == 0 ? r : 2 * r + c;
    }
    const int u = k - flush_group_bottom(D);  // node of the group's upper subtree, heap order
    if (u < 0 || u >= GS - 1) return -1;
    const int l = ilog2(u + 1);          // level of u within the group's subtree
    const int lg = D - 2 - ilog2(GS) + l;  // its level in the tree
    return (1 << lg) - 1 + g * (1 << l) + (u - ((1 << l) - 1));
}

static_assert(flush_batches(8) <= 64, "batch flags are one 64-bit word per tree");

// Everything of a tree that the consumer kernel stages, but its line maps, as 16-byte words
// (copied asynchronously, no registers), in chunks of a whole tree, at depth 8 of a unit: the units'
// nodes; the phi offset (feature x row stride of the phi tile) of every flush position,
// 16 bits; with several units those of the tree's last batch, the nodes above the units; per
// unit a word of flags, live subtrees in bits 0-7, flush (no repeated feature) and real of its
// batches and the last batch in bits 8-15 and 16-23; per batch the positions whose feature an
// earlier position of the batch has (0xFF when they repeat among themselves).  After the
// chunks, with several levels above the units, the nodes of those.  The offsets depend on the
// tile's rows, so an ensemble has an image of its trees for every tile size (one of wide tiles,
// k_explain.cuh, only theirs).
WDF_HD constexpr int chunk_units(int D) { return D == 8 ? 1 : units_per_tree(D); }
WDF_HD constexpr int tree_chunks(int D) { return units_per_tree(D) / chunk_units(D); }
WDF_HD constexpr int chunk_positions(int D) {
    return chunk_units(D) * flush_group_len(D) + (units_per_tree(D) > 1 ? 8 : 0);
}
WDF_HD constexpr int chunk_offsets(int D) { return chunk_units(D) * 32 * (int)sizeof(UnitNode); }
WDF_HD constexpr int chunk_flags(int D) { return chunk_offsets(D) + 2 * chunk_positions(D); }
WDF_HD constexpr int chunk_repeats(int D) { return chunk_flags(D) + 4 * chunk_units(D); }
WDF_HD constexpr int chunk_bytes(int D) { return (chunk_repeats(D) + chunk_positions(D) / 8 + 15) & ~15; }
WDF_HD constexpr int image_top(int D) { return tree_chunks(D) * chunk_bytes(D); }
WDF_HD constexpr int image_bytes(int D) { return image_top(D) + (unit_top(D) > 1 ? 8 * (int)sizeof(UnitNode) : 0); }
static_assert(flush_group_len(8) / 8 < 8 && image_bytes(8) % 16 == 0, "chunk layout");
// A row's phi is the sum of the sums of its ensemble's parts, in part order: part p of P holds
// trees [T p / P, T (p + 1) / P), each part's nodes added in the consumer kernel's order from
// zero.  The split depends on the ensemble alone, so a row's result does not depend on how
// many blocks share its parts.  About 50 trees of depth 6 to a part: a part's end costs what
// 1.3 such trees cost.
WDF_HD inline int explain_parts(int T, int D) {
    const long long p = (((long long)T << D) + 1600) / 3200;
    return p < 1 ? 1 : p > 8 ? 8 : (int)p;
}

constexpr int kImages = 3;
WDF_HD constexpr int image_rows(int i) { return 32 << i; }  // tile rows of image i

}  // namespace wdf
