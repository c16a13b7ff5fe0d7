// Background side of Algorithm 3, step 1: decision patterns of every background row
// (Algorithm 1, kept in registers) and their counts vc[l][p_b] (Eq.
// "bg_shap_derivation" step (d)); plus the per-leaf marginals and E_b f(b).
//
// The joint entry e = (pattern at a bottom subtree's root, the three decisions inside the
// subtree) of every background row is counted per tree and live bottom subtree; the four leaf
// patterns of the subtree are functions of e, so per-leaf counts are exact marginals of
// these joint counts (the sibling-leaf observation of section "Algorithmic Improvements"
// item 3, applied two levels up).
#include <algorithm>
#include <cmath>

#include "launch.h"
#include "wdf_device.cuh"

namespace wdf {

// Depth <= 6: counting on the tensor cores.  A joint count is a sum over rows of products of indicators:
// count(R, n) = sum_rows [ancestor decisions = R] [subtree decisions = n], so 16 ancestor
// patterns x 8 subtree patterns of one bottom subtree are a small matrix product over rows
// with operands built in registers from the rows' decision bits.  A warp owns one unit
// (tree_layout.h) and keeps all its counters in registers; no counter is touched in memory
// until the block's rows are done.
//
// Per tile of 128 rows a warp
//   - evaluates its unit's 31 nodes, lane = node, for 32 rows at a time on the sliced codes
//     (two or three 16-byte shared loads and 8 or 12 logic instructions per 32 x 32 decisions;
//     the rank masks stay in registers for the whole launch) and exchanges the decision
//     words through shared memory: lane (g, q) = (lane / 4, lane % 4) needs all nodes' words
//     of row block q, the rows its MMA fragments cover;
//   - forms the indicator words: ancestor pattern g (and g + 8, for the MMA's upper rows)
//     per sibling pair of subtrees, which share their ancestors, and subtree pattern g;
//   - expands each word into eight FP16-pair registers, two rows per FP16 value, so that four
//     m16n8k16 MMAs cover the tile (depth 6's sixteen ancestor patterns are one m16).  An FP16 value with only bits 0..10 set is that integer
//     times 2^-24.  The ancestor side keeps bits j and j + 8 of each half (one AND, the shift
//     shared by three registers); the subtree side, whose words are stored with the bits of
//     each half reversed, puts the same two rows at bits 10 - j and 2 - j.  Every product is
//     then 2^10 (a b + a' b') + 2^2 a b' + 2^18 a' b, in units of 2^-48: the wanted sum over
//     the tile (at most 128) and the two cross sums (at most 64) are separate bytes of the
//     FP32 accumulator, which starts from 2^-23 so that its mantissa is their integer;
//   - adds the middle byte of every accumulator to an integer counter.
// E4M3, 8-bit integer and 1-bit MMAs are emulated here (20, 17 and 142 issue slots per
// instruction); one row per FP16 value takes twice the MMAs and nearly twice the logic.
// Bound by the logic pipe (58 % busy, issue 55 %): 2.31 ms per 1M rows and 200 trees of depth 6,
// where one shared-memory atomic per (row, bottom subtree), each row's decisions made node by
// node, took 5.14 ms, and k_bg_add below takes 20 % more (depth 5: 12 %).
template <int D>
struct Unit {
    static constexpr int H = unit_height(D), TOP = unit_top(D), UPT = units_per_tree(D);
    static constexpr int NLOC = (1 << H) - 1, NSU = 1 << (H - 2);  // nodes and bottom subtrees
};
constexpr int kCountWarps = 16;  // of an SM (k_bg_count's registers)
constexpr int kDecStride = 36;  // words of a row block's decision words: 9 * 16 bytes, so that the
                                // four row blocks of a fragment lie in different banks

constexpr float kCountBase = 0x1p-23f;  // an accumulator with all three sums zero

__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1, const float *c) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// A word and its shifts by 3 and 6, so that rows j and j + 8 of each half are bits i and i + 8
// (i = j % 3) of shift j / 3.
struct Shifts {
    uint32_t w[3];
    __device__ __forceinline__ void set(uint32_t x) {
        w[0] = x; w[1] = (x >> 3); w[2] = (x >> 6);
    }
};
// Register j: rows j and j + 8 of each half of x & y, at bits i and i + 8.
__device__ __forceinline__ void expand_a(const Shifts &x, const Shifts &y, uint32_t (&r)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) r[j] = x.w[j / 3] & y.w[j / 3] & (0x01010101u << (j % 3));
}
// The same rows, from a word with each half's bits reversed, at bits 10 - i and 2 - i.
__device__ __forceinline__ void expand_b(uint32_t y, uint32_t (&r)[8]) {
    const uint32_t y0 = (y >> 5), y3 = (y >> 2), y6 = y << 1;
#pragma unroll
    for (int j = 0; j < 8; ++j) r[j] = (j < 3 ? y0 : j < 6 ? y3 : y6) & (0x01010101u << (2 - j % 3));
}

// The decision words of one node for the row blocks of a tile.
struct SliceNode {
    uint32_t at, m[3][4];
    __device__ __forceinline__ void load(const UnitNode *p) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
        at = v.x;
#pragma unroll
        for (int k = 0; k < 3; ++k) rank_masks(v.y, k, m[k]);
    }
    __device__ __forceinline__ uint32_t decide1(const uint4 *block, const SliceArrays &sa) const {
        const int col = unit_column(at), nq = unit_quads(at);
        uint32_t w = 0u - unit_start(at);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k < nq) w = slice_le(w, block[sa.qbase[k] + col], m[k]);
        return w;
    }
    template <int N>
    __device__ __forceinline__ void decide(const uint4 *tile, const SliceArrays &sa, uint32_t (&w)[N]) const {
        const int col = unit_column(at), nq = unit_quads(at);
        const uint32_t le0 = 0u - unit_start(at);
#pragma unroll
        for (int b = 0; b < N; ++b) w[b] = le0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (k < nq) {
                uint4 q[N];
#pragma unroll
                for (int b = 0; b < N; ++b) q[b] = tile[b * sa.quads + sa.qbase[k] + col];
#pragma unroll
                for (int b = 0; b < N; ++b) w[b] = slice_le(w[b], q[b], m[k]);
            }
        }
    }
};

// codes: rows [0, m) of one encoded chunk, padded to a multiple of 128 rows.  Block (chunk,
// slice): units [chunk * W, ...), one per warp, over the tiles of 128 rows slice, slice +
// nslices, ... in runs of SUB tiles.  STAGES runs in shared memory, filled by cp.async ahead
// of their use (a barrier per run); STAGES = 0 reads the codes from global memory (rows too wide for two tiles).
template <int D, int STAGES, int SUB>
__global__ void __launch_bounds__(32 * kCountWarps, 1) k_bg_count(const unsigned char *__restrict__ codes, int64_t m,
                                                                   SliceArrays sa, const TreeMeta *__restrict__ meta,
                                                                   int units, int chunks, uint32_t *__restrict__ hist) {
    using S = Shape<D>;
    using N = Unit<D>;
    static_assert(N::TOP <= 1, "one m16 of ancestor patterns");
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    const int chunk = blockIdx.x % chunks, slice = blockIdx.x / chunks, nslices = gridDim.x / chunks;
    const int unit = min(chunk * W + warp, units - 1);  // a spare warp repeats the last unit and adds nothing
    const int t = unit / N::UPT, u = unit % N::UPT;
    const int tile16 = 4 * sa.quads, run16 = SUB * tile16;  // 16-byte words of a tile, of a run
    uint4 *ring = reinterpret_cast<uint4 *>(smem_raw);
    uint32_t *dec = reinterpret_cast<uint32_t *>(smem_raw + (size_t)STAGES * run16 * 16) + warp * 4 * kDecStride;
    const int64_t tiles = (m + kBgTileRows - 1) / kBgTileRows, runs = (tiles + SUB - 1) / SUB;

    SliceNode node;
    {
        const UnitNode *un = sa.unit + (size_t)unit * 32 + lane;
        if (N::TOP > 0 && lane == 31) un = sa.unit + (size_t)t * N::UPT * 32 + 31;  // the root
        node.load(un);
    }
    const uint32_t live = (uint32_t)(__ldg(&meta[t].live) >> (u * N::NSU)) & ((1u << N::NSU) - 1u);
    const bool flip = lane >= N::NSU - 1 && lane < N::NLOC;  // nodes of a bottom subtree
    const int g = lane >> 2, q = lane & 3;
    const uint32_t x0 = (g & 4) ? 0u : ~0u, x1 = (g & 2) ? 0u : ~0u, x2 = (g & 1) ? 0u : ~0u;
    uint32_t count[N::NSU][4];
#pragma unroll
    for (int s = 0; s < N::NSU; ++s)
#pragma unroll
        for (int k = 0; k < 4; ++k) count[s][k] = 0u;

    const float base[4] = {kCountBase, kCountBase, kCountBase, kCountBase};
    auto fetch = [&](int64_t run, int stage) {
        if constexpr (STAGES > 0) {
            if (run < runs) {
                const int n = (int)min((int64_t)SUB, tiles - run * SUB) * tile16;
                const uint4 *src = reinterpret_cast<const uint4 *>(codes) + run * run16 + tid;
                uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + (size_t)stage * run16 + tid);
                for (int i = tid; i < n; i += blockDim.x, src += blockDim.x, dst += 16u * blockDim.x)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
            }
            asm volatile("cp.async.commit_group;");
        }
    };
#pragma unroll
    for (int k = 0; k + 1 < STAGES; ++k) fetch(slice + (int64_t)k * nslices, k);
    int stage = 0;
    for (int64_t run = slice; run < runs; run += nslices) {
        const uint4 *src;
        if constexpr (STAGES > 0) {
            asm volatile("cp.async.wait_group %0;" ::"n"(STAGES > 1 ? STAGES - 2 : 0));
            __syncthreads();
            const int into = stage == 0 ? STAGES - 1 : stage - 1;
            fetch(run + (int64_t)(STAGES - 1) * nslices, into);
            src = ring + (size_t)stage * run16;
            stage = stage + 1 == STAGES ? 0 : stage + 1;
        } else {
            src = reinterpret_cast<const uint4 *>(codes) + run * run16;
        }
        const int here = (int)min((int64_t)SUB, tiles - run * SUB);
        int left = (int)min(m - run * SUB * kBgTileRows, (int64_t)(1 << 30)) - 32 * q;  // rows from row block q on
#pragma unroll 1
        for (int sub = 0; sub < here; ++sub, src += tile16, left -= kBgTileRows) {
            uint32_t w[4];
            node.decide(src, sa, w);
#pragma unroll
            for (int b = 0; b < 4; ++b) dec[b * kDecStride + lane] = flip ? __byte_perm(__brev(w[b]), 0u, 0x1032) : w[b];
            __syncwarp();
            constexpr int NV = (N::NLOC + 3) / 4;
            uint32_t d[4 * NV > 32 ? 4 * NV : 32];
            const uint32_t *mine = dec + q * kDecStride;
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const uint4 v = reinterpret_cast<const uint4 *>(mine)[i];
                d[4 * i] = v.x; d[4 * i + 1] = v.y; d[4 * i + 2] = v.z; d[4 * i + 3] = v.w;
            }
            __syncwarp();
            const uint32_t valid = left >= 32 ? ~0u : (left > 0 ? (1u << left) - 1u : 0u);
            // depth 6: rows that the root sends right and left
            Shifts in[1 << N::TOP];
            in[0].set(N::TOP > 0 ? valid & ~d[31] : valid);
            if constexpr (N::TOP > 0) in[1].set(valid & d[31]);
            constexpr int NP = N::NSU > 1 ? N::NSU / 2 : 1;  // sibling pairs
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                // the pair's ancestors inside the unit: the last three decisions of the pattern
                uint32_t anc = ~0u;
                if constexpr (N::H == 5) anc = (d[0] ^ x0) & (d[1 + (j >> 1)] ^ x1) & (d[3 + j] ^ x2);
                if constexpr (N::H == 4) anc = (d[0] ^ x1) & (d[1 + j] ^ x2);
                if constexpr (N::H == 3) anc = d[0] ^ x2;
                Shifts own;
                own.set(anc);
                uint32_t rb[2][8];
#pragma unroll
                for (int h = 0; h < (N::NSU > 1 ? 2 : 1); ++h) {
                    const int c = N::NSU - 1 + 3 * (2 * j + h);  // the root's left child, right child and the root
                    expand_b((d[c + 2] ^ x0) & (d[c + 1] ^ x1) & (d[c] ^ x2), rb[h]);
                }
                uint32_t ra[2][8];
                expand_a(own, in[0], ra[0]);
                if constexpr (N::TOP > 0) expand_a(own, in[1], ra[1]);
                float acc[2][4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int h = 0; h < (N::NSU > 1 ? 2 : 1); ++h)
                        mma_f16(acc[h], ra[0][2 * k], N::TOP > 0 ? ra[1][2 * k] : 0u, ra[0][2 * k + 1],
                                N::TOP > 0 ? ra[1][2 * k + 1] : 0u, rb[h][2 * k], rb[h][2 * k + 1],
                                k == 0 ? base : acc[h]);
#pragma unroll
                for (int h = 0; h < (N::NSU > 1 ? 2 : 1); ++h)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        count[2 * j + h][k] = __dp4a(__float_as_uint(acc[h][k]), 0x00000100u, count[2 * j + h][k]);
            }
        }
    }
    if (chunk * W + warp >= units) return;
#pragma unroll
    for (int s = 0; s < N::NSU; ++s) {
        if (!((live >> s) & 1u)) continue;
        uint32_t *h = hist + ((size_t)t * S::NS + u * N::NSU + s) * S::E;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // accumulator k: pattern row g (+ 8 for k >= 2), subtree pattern 2q + (k & 1)
            const uint32_t R = (uint32_t)g + 8u * (k >> 1);
            const uint32_t c = count[s][k];
            if (R < (uint32_t)(S::E >> 3) && c) atomicAdd(h + ((R << 3) | (2 * q + (k & 1))), c);
        }
    }
}

// Warps (units) per block and row slices of a launch: all blocks resident, one or more per
// SM, and the busiest SM's warps x tiles as few as possible (a block also spends about
// two tiles' worth on loading its nodes and adding its counters; fewer than 3/4 of the
// warps an SM can hold take as long as that many).  On a tie the smaller blocks, which wait
// less at their barriers.
template <int D, int STAGES, int SUB>
static cudaError_t bg_count_t(const unsigned char *codes, int64_t m, const SliceArrays &sa, const TreeMeta *meta, int T,
                              uint32_t *hist, const DevInfo &dev, cudaStream_t st) {
    using N = Unit<D>;
    const int units = T * N::UPT;
    const int64_t runs = ((m + kBgTileRows - 1) / kBgTileRows + SUB - 1) / SUB;
    auto smem = [&](int W) { return (size_t)STAGES * SUB * sa.quads * 64 + (size_t)W * 4 * kDecStride * 4; };
    int64_t best = -1, best_slices = 1;
    int best_w = 1;
    for (int W = std::min(units, kCountWarps); W >= 1; --W) {
        const int64_t chunks = (units + W - 1) / W;
        const int64_t per_sm = std::max<int64_t>(
            1, std::min<int64_t>(kCountWarps / W, (int64_t)(dev.smem_optin / (smem(W) + 1024))));
        const int64_t slices = std::max<int64_t>(1, std::min<int64_t>(runs, dev.sms * per_sm / chunks));
        const int64_t waves = (chunks * slices + dev.sms * per_sm - 1) / (dev.sms * per_sm);
        const int64_t warps = W * std::min(per_sm, (chunks * slices + dev.sms - 1) / dev.sms);  // of one SM
        const int64_t cost = waves * std::max<int64_t>(warps, 3 * kCountWarps / 4) * (((runs + slices - 1) / slices) * SUB + 2);
        if (best < 0 || cost <= best) {
            best = cost;
            best_w = W;
            best_slices = slices;
        }
    }
    const int chunks = (units + best_w - 1) / best_w;
    auto kern = k_bg_count<D, STAGES, SUB>;
    cudaError_t err = allow_shared(kern, smem(best_w), dev);
    if (err != cudaSuccess) return err;
    kern<<<(unsigned)(best_slices * chunks), 32 * best_w, smem(best_w), st>>>(codes, m, sa, meta, units, chunks, hist);
    count_launches(1);
    return cudaGetLastError();
}

// Depth 7 and 8: counting by shared-memory atomics (a unit's 8 x 2^(D+1) counters grow with the
// depth, and with them the MMAs, but not a row's 8 entries per unit).  Two warps own one unit and
// its counters in shared memory, each takes two of a tile's four row blocks.  A warp evaluates
// the unit's nodes on the sliced codes as above, turns the words of 32 rows so that each lane
// has its row's 31 decisions (wdf_device.cuh), and adds one to the row's entry of every live
// subtree.  Latency-bound (issue 53 %, shared-memory wavefronts 60 %, 5.6 of them per atomic);
// four warps per unit with one row block each take 15 % longer, one warp with four 7 %.
// 60,013 rows and 300 trees of depth 8 2.48 -> 1.44 ms, 60,000 rows and 300 trees of depth 7 0.77
// -> 0.66 (from MMAs with four and two m16 tiles of ancestor patterns), encoding included.
template <int D, int STAGES>
__global__ void __launch_bounds__(512, 1) k_bg_add(const unsigned char *__restrict__ codes, int64_t m, SliceArrays sa,
                                                  const TreeMeta *__restrict__ meta, int units, int chunks,
                                                  uint32_t *__restrict__ hist) {
    using S = Shape<D>;
    using N = Unit<D>;
    constexpr int GS = N::NSU, TOP = N::TOP, CELLS = GS * S::E;
    static_assert(N::H == 5 && CELLS % 8 == 0, "units of 31 nodes, counters in whole 32 bytes");
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 6, half = (tid >> 5) & 1, W = blockDim.x >> 6;
    const int chunk = blockIdx.x % chunks, slice = blockIdx.x / chunks, nslices = gridDim.x / chunks;
    const bool spare = chunk * W + warp >= units;
    const int unit = min(chunk * W + warp, units - 1), t = unit / N::UPT, u = unit % N::UPT;
    const int tile16 = 4 * sa.quads;  // 16-byte words of a tile
    uint4 *ring = reinterpret_cast<uint4 *>(smem_raw);
    uint32_t *cells = reinterpret_cast<uint32_t *>(smem_raw + (size_t)STAGES * tile16 * 16) + warp * CELLS;
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(cells);
    const int64_t tiles = (m + kBgTileRows - 1) / kBgTileRows;

    SliceNode node, top;  // as in k_bg_count
    {
        const UnitNode *un = sa.unit + (size_t)unit * 32 + lane;
        if (TOP > 0 && lane == 31) un = sa.unit + (size_t)t * N::UPT * 32 + 31;  // the root
        node.load(un);
        if constexpr (TOP > 1) {
            const int k = min(1 + (lane >> 1), TOP - 1), v = (1 << k) - 1 + (u >> (TOP - k));
            top.load(sa.unit + ((size_t)t * N::UPT + v) * 32 + 31);
        }
    }
    const uint32_t live = spare ? 0u : (uint32_t)(__ldg(&meta[t].live) >> (u * GS)) & ((1u << GS) - 1u);
    for (int i = tid; i < W * CELLS; i += blockDim.x)
        reinterpret_cast<uint32_t *>(smem_raw + (size_t)STAGES * tile16 * 16)[i] = 0u;
    __syncthreads();

    auto fetch = [&](int64_t tile, int stage) {
        if constexpr (STAGES > 0) {
            if (tile < tiles) {
                const uint4 *src = reinterpret_cast<const uint4 *>(codes) + tile * tile16 + tid;
                uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + (size_t)stage * tile16 + tid);
                for (int i = tid; i < tile16; i += blockDim.x, src += blockDim.x, dst += 16u * blockDim.x)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
            }
            asm volatile("cp.async.commit_group;");
        }
    };
#pragma unroll
    for (int k = 0; k + 1 < STAGES; ++k) fetch(slice + (int64_t)k * nslices, k);
    int stage = 0;
    for (int64_t tile = slice; tile < tiles; tile += nslices) {
        const uint4 *src;
        if constexpr (STAGES > 0) {
            asm volatile("cp.async.wait_group %0;" ::"n"(STAGES > 1 ? STAGES - 2 : 0));
            __syncthreads();
            fetch(tile + (int64_t)(STAGES - 1) * nslices, stage == 0 ? STAGES - 1 : stage - 1);
            src = ring + (size_t)stage * tile16;
            stage = stage + 1 == STAGES ? 0 : stage + 1;
        } else {
            src = reinterpret_cast<const uint4 *>(codes) + tile * tile16;
        }
        src += 2 * half * sa.quads;
        const int left = (int)min(m - tile * kBgTileRows, (int64_t)kBgTileRows) - 64 * half;  // rows of this warp
        uint32_t w[2], tw = 0u;
        node.decide(src, sa, w);
        if constexpr (TOP > 1) {
            if (lane < 2 * (TOP - 1)) tw = top.decide1(src + (lane & 1) * sa.quads, sa);
        }
        transpose32(w, lane);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            uint32_t path = TOP > 0 ? w[b] >> 31 : 0u;
#pragma unroll
            for (int k = 1; k < TOP; ++k) path = 2u * path + ((__shfl_sync(0xFFFFFFFFu, tw, 2 * (k - 1) + b) >> lane) & 1u);
            // byte offsets, entry e of subtree j at 4 (j E + e): R of the children of the unit's
            // nodes above its subtrees, 32 bytes (eight entries) apart; the entry's own bits are ORed
            // in below, so the counters lie on a 32-byte boundary (the array does, and so many tiles
            // and units into it)
            uint32_t R[GS - 1];
            R[0] = 64u * path | ((w[b] << 5) & 32u);
#pragma unroll
            for (int k = 1; k < GS - 1; ++k) {
                R[k] = 2u * R[(k - 1) >> 1] | ((k < 5 ? w[b] << (5 - k) : w[b] >> (k - 5)) & 32u);
            }
#pragma unroll
            for (int k = GS / 2 - 1; k < GS - 1; ++k) R[k] += at;
            if (32 * b + lane < left) {
#pragma unroll
                for (int j = 0; j < GS; ++j)
                    if ((live >> j) & 1u)  // the same for all lanes
                        asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(
                                         (((w[b] >> (GS - 3 + 3 * j)) & 28u) | R[(GS - 2 + j) >> 1]) + 4u * j * S::E)
                                     : "memory");
            }
        }
    }
    __syncthreads();
    if (spare) return;
    uint32_t *h = hist + ((size_t)t * S::NS + u * GS) * S::E;
    for (int i = (tid & 63); i < CELLS; i += 64) {
        const uint32_t c = cells[i];
        if (c) atomicAdd(h + i, c);
    }
}

// Eight units per block (as many as fit) and the number of row slices with the least time by
// this measure: a block takes its tiles' time and four tiles' more for its counters; blocks go
// round the SMs; they differ in live subtrees, so a round ends 14 % of a block's time late.
// 300 trees, 60,000 rows: depth 8, 1, 2 and 3 slices 1.54, 1.46 and 1.43 ms; depth 7, 1, 2, 4
// and 6 slices 709, 684, 655 and 648 us.
constexpr int kAddUnits = 8;
template <int D, int STAGES>
static cudaError_t bg_add_t(const unsigned char *codes, int64_t m, const SliceArrays &sa, const TreeMeta *meta, int T,
                            int W, uint32_t *hist, const DevInfo &dev, cudaStream_t st) {
    const int units = T * Unit<D>::UPT, chunks = (units + W - 1) / W;
    const int64_t tiles = (m + kBgTileRows - 1) / kBgTileRows;
    int64_t slices = 1;
    double least = 0.0;
    for (int64_t s = 1; s <= std::min<int64_t>(tiles, 64); ++s) {
        const double one = (double)((tiles + s - 1) / s + 4), rounds = (double)(chunks * s) / dev.sms;
        const double cost = one * (0.14 + (rounds <= 1.0 ? 1.0 : 0.5 * (rounds + std::ceil(rounds))));
        if (s == 1 || cost < least) {
            slices = s;
            least = cost;
        }
    }
    const size_t smem = (size_t)STAGES * sa.quads * 64 + (size_t)W * Unit<D>::NSU * Shape<D>::E * 4;
    auto kern = k_bg_add<D, STAGES>;
    cudaError_t err = allow_shared(kern, smem, dev);
    if (err != cudaSuccess) return err;
    kern<<<(unsigned)(slices * chunks), 64 * W, smem, st>>>(codes, m, sa, meta, units, chunks, hist);
    count_launches(1);
    return cudaGetLastError();
}

// Long chunks of rows run with four tiles per barrier, where three such runs fit: 2.31 ms per
// 1M rows and 200 depth-6 trees against 2.53 with two tiles per run and two half-size blocks
// per SM (the warps of a block drift apart and wait at every barrier).  Below 16,384 rows a
// block would get too few runs to share evenly.
constexpr int64_t kBgLongRows = 16384;
template <int D>
static cudaError_t bg_count(const unsigned char *codes, int64_t m, const SliceArrays &sa, const TreeMeta *meta, int T,
                            uint32_t *hist, const DevInfo &dev, cudaStream_t st) {
    if constexpr (D >= 7) {
        // rows too wide for two tiles beside four units' counters are read from global memory
        const size_t unit = (size_t)Unit<D>::NSU * Shape<D>::E * 4, ring = (size_t)2 * sa.quads * 64;
        const int most = std::min(kAddUnits, T * Unit<D>::UPT);
        const int fit = ring < dev.smem_optin ? (int)std::min<size_t>(most, (dev.smem_optin - ring) / unit) : 0;
        if (fit >= std::min(most, 4)) return bg_add_t<D, 2>(codes, m, sa, meta, T, fit, hist, dev, st);
        return bg_add_t<D, 0>(codes, m, sa, meta, T, most, hist, dev, st);
    } else {
        const size_t dec = (size_t)kCountWarps * 4 * kDecStride * 4;
        if (3 * 4 * (size_t)sa.quads * 64 + dec <= dev.smem_optin && m >= kBgLongRows)
            return bg_count_t<D, 3, 4>(codes, m, sa, meta, T, hist, dev, st);
        if (3 * (size_t)sa.quads * 64 + dec <= dev.smem_optin)
            return bg_count_t<D, 3, 1>(codes, m, sa, meta, T, hist, dev, st);
        return bg_count_t<D, 0, 1>(codes, m, sa, meta, T, hist, dev, st);
    }
}

cudaError_t launch_bg_hist(int D, const float *B, int64_t m, int64_t ldb, const TreeMeta *meta, const SliceArrays &sa,
                           int T, unsigned char *codes, int64_t code_rows, uint32_t *hist, const DevInfo &dev,
                           cudaStream_t st, const BgOverlap *ov) {
    if (m == 0) return cudaSuccess;
    if (code_rows < kBgTileRows || code_rows % kBgTileRows) return cudaErrorInvalidValue;
    cudaError_t err = cudaSuccess;
    if (ov) {
        // the side stream starts after everything already queued on st (B, the zeroed counts)
        err = cudaEventRecord(ov->cnt[0], st);
        if (err == cudaSuccess) err = cudaStreamWaitEvent(ov->side, ov->cnt[0], 0);
        if (err != cudaSuccess) return err;
    }
    int64_t k = 0;
    for (int64_t r0 = 0; r0 < m; r0 += code_rows, ++k) {
        const int64_t rows = std::min(code_rows, m - r0);
        const int64_t rows_pad = (rows + kBgTileRows - 1) / kBgTileRows * kBgTileRows;
        const int b = ov ? (int)(k & 1) : 0;
        unsigned char *buf = b ? ov->codes1 : codes;
        if (ov) {
            // encode chunk k on the side stream once the count of chunk k - 2 (the last
            // reader of this buffer) is done; the count of chunk k waits for the encode
            if (k >= 2) err = cudaStreamWaitEvent(ov->side, ov->cnt[b], 0);
            if (err == cudaSuccess) err = launch_encode_slices(B + r0 * ldb, rows, ldb, sa, rows_pad, buf, dev, ov->side);
            if (err == cudaSuccess) err = cudaEventRecord(ov->enc[b], ov->side);
            if (err == cudaSuccess) err = cudaStreamWaitEvent(st, ov->enc[b], 0);
        } else {
            err = launch_encode_slices(B + r0 * ldb, rows, ldb, sa, rows_pad, buf, dev, st);
        }
        if (err != cudaSuccess) return err;
        switch (D) {
            case 2: err = bg_count<2>(buf, rows, sa, meta, T, hist, dev, st); break;
            case 3: err = bg_count<3>(buf, rows, sa, meta, T, hist, dev, st); break;
            case 4: err = bg_count<4>(buf, rows, sa, meta, T, hist, dev, st); break;
            case 5: err = bg_count<5>(buf, rows, sa, meta, T, hist, dev, st); break;
            case 6: err = bg_count<6>(buf, rows, sa, meta, T, hist, dev, st); break;
            case 7: err = bg_count<7>(buf, rows, sa, meta, T, hist, dev, st); break;
            case 8: err = bg_count<8>(buf, rows, sa, meta, T, hist, dev, st); break;
            default: return cudaErrorInvalidValue;
        }
        if (err == cudaSuccess && ov) err = cudaEventRecord(ov->cnt[b], st);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

// vc[row][p] of every live leaf row; A (when non-null) receives the counts as FP32, the A
// operand of the contraction (exact below 2^24 background rows).
__global__ void k_leaf_counts(int D, const uint32_t *__restrict__ hist, const int32_t *__restrict__ group_leaf,
                              int n_live, uint32_t *__restrict__ vc, float *__restrict__ A) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)n_live << D) return;
    const uint32_t v = leaf_count(D, hist, __ldg(group_leaf + (idx >> D)), (uint32_t)(idx & ((1 << D) - 1)));
    if (vc) vc[idx] = v;
    if (A) A[idx] = (float)v;
}

cudaError_t launch_leaf_counts(int D, const uint32_t *hist, const int32_t *group_leaf, int n_live, uint32_t *vc,
                               float *A, cudaStream_t st) {
    const int64_t total = (int64_t)n_live << D;
    if (total == 0) return cudaSuccess;
    const int threads = 256;
    k_leaf_counts<<<(unsigned)((total + threads - 1) / threads), threads, 0, st>>>(D, hist, group_leaf, n_live, vc,
                                                                                  A);
    count_launches(1);
    return cudaGetLastError();
}

// Path-dependent frequencies (Eq. "path_dependent_estimation"): for live leaf row `row`
// with cover ratios r_k = cover(path node k+1) / cover(path node k), the frequency of
// baseline pattern p is the product over the path of r_k where bit D-1-k of p is 1 and
// of 1 - r_k where it is 0, in FP64, stored as the FP32 A operand.
__global__ void k_pd_freq(int D, const double *__restrict__ ratio, int n_live, float *__restrict__ A) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= ((int64_t)n_live << D)) return;
    const int row = (int)(idx >> D);
    const uint32_t p = (uint32_t)(idx & ((1 << D) - 1));
    double f = 1.0;
    for (int k = 0; k < D; ++k) {
        const double r = __ldg(ratio + (size_t)row * D + k);
        f *= ((p >> (D - 1 - k)) & 1u) ? r : 1.0 - r;
    }
    A[idx] = (float)f;
}

cudaError_t launch_pd_freq(int D, const double *ratio, int n_live, float *A, cudaStream_t st) {
    const int64_t total = (int64_t)n_live << D;
    if (total == 0) return cudaSuccess;
    k_pd_freq<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(D, ratio, n_live, A);
    count_launches(1);
    return cudaGetLastError();
}

// v({}) = sum_l w_l * freq_l(all ones): for the background game freq = count / m (a row
// reaches leaf l exactly when its pattern there is all ones, so this is E_b f(b)); for
// the path-dependent game (ratio non-null) freq = the product of the leaf's cover ratios.
// kBaseBlocks blocks each add the leaves block, block + kBaseBlocks, ... of 256 in a fixed
// order, one more adds the blocks' sums: 14 us for 41,000 leaves of depth 8, where one block
// alone took 300, waiting for one load after another.
__device__ __forceinline__ double block_sum(double x, double *red) {
    red[threadIdx.x] = x;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    return red[0];
}

__global__ void __launch_bounds__(256) k_base_partial(int D, const uint32_t *__restrict__ hist,
                                                      const int32_t *__restrict__ group_leaf,
                                                      const double *__restrict__ ratio, const double *__restrict__ w,
                                                      int n_live, int64_t m, double *__restrict__ out) {
    __shared__ double red[256];
    double acc = 0.0;
    for (int r = blockIdx.x * 256 + threadIdx.x; r < n_live; r += kBaseBlocks * 256) {
        double f;
        if (ratio) {
            f = 1.0;
            for (int k = 0; k < D; ++k) f *= ratio[(size_t)r * D + k];
        } else {
            f = (double)leaf_count(D, hist, __ldg(group_leaf + r), (1u << D) - 1u) / (double)m;
        }
        acc += w[r] * f;
    }
    const double sum = block_sum(acc, red);
    if (threadIdx.x == 0) out[1 + blockIdx.x] = sum;
}

__global__ void __launch_bounds__(kBaseBlocks) k_base_final(double *__restrict__ out) {
    __shared__ double red[kBaseBlocks];
    const double sum = block_sum(out[1 + threadIdx.x], red);
    if (threadIdx.x == 0) out[0] = sum;
}

cudaError_t launch_base_value(int D, const uint32_t *hist, const int32_t *group_leaf, const double *ratio,
                              const double *leaf_w_rows, int n_live, int64_t m, double *out, cudaStream_t st) {
    k_base_partial<<<kBaseBlocks, 256, 0, st>>>(D, hist, group_leaf, ratio, leaf_w_rows, n_live, m, out);
    k_base_final<<<1, kBaseBlocks, 0, st>>>(out);
    count_launches(2);
    return cudaGetLastError();
}

// scale[row] = w_row / m, the leaf weight and the 1/|B| of Eq. "bg_shap_derivation"
// step (e) folded into one FP32 factor per leaf.
__global__ void k_scale(const double *__restrict__ w, int n_live, int64_t m, float *__restrict__ scale) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_live) scale[i] = (float)(w[i] / (double)m);
}

cudaError_t launch_scale(const double *w, int n_live, int64_t m, float *scale, cudaStream_t st) {
    if (n_live == 0) return cudaSuccess;
    k_scale<<<(n_live + 255) / 256, 256, 0, st>>>(w, n_live, m, scale);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace wdf
