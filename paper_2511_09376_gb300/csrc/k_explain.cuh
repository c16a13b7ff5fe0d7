// Consumer side of Algorithm 3, step 4 (Eq. "bg_shap_derivation" step (g)):
// phi[c, i] = sum over trees and leaves of s_{l,i}[P[l][c]].
//
// A block takes a tile of consumer rows, two warps per 32 rows, a lane per row.  It stages its rows' sliced
// decision codes (tree_layout.h) in shared memory together with a per-row phi accumulator
// (feature-major) and walks the trees.  Per unit of a tree (31 nodes, eight bottom subtrees)
// each warp
//   - evaluates the unit's nodes for its 32 rows, lane = node: two or three 16-byte shared
//     loads and eight or twelve logic instructions for 32 x 32 decisions, then a 32 x 32 bit
//     transpose leaves every lane with its own row's decisions (evaluating them node by
//     node, lane = row, took two shared loads and four instructions per node);
//   - forms the row's entry at every bottom subtree and gathers one slot vector per subtree
//     from the folded table, all of a unit's gathers in flight together;
//   - sums the slots of the nodes above the bottom subtrees in registers and adds every
//     node's value into phi[feature of the node] in the fixed flush order of tree_layout.h, a
//     batch at a time: a batch that repeats no feature reads its phi values before writing
//     any, so the shared-memory round trips overlap; another batch adds its features' first
//     positions so and the repeats after them (one by one where they repeat among themselves).
//     Pass-through nodes add into a scratch row, a batch of pass-through nodes only is
//     skipped.
// The trees come in parts (explain_parts): a part's sums start from zero and are added to
// the row's phi at its end.  The order of every floating-point addition into a row's phi
// depends only on the ensemble, never on which rows share a block.
//
// Per row and depth-6 tree: about 13 32-byte gathers (four 128-byte lines per quarter warp) and
// 50 phi read-modify-writes, some 430 L1 data-pipe wavefronts per warp and tree.  10.2 ms per 1M
// rows and 200 trees of depth 6 (127 features), 515 SM clocks per warp and tree of 32 rows (L1
// pipe 81 %), 546 while its gathers allocated in the L1 cache; of that form, one warp per 32
// rows took 677 (two units' gathers in flight, ten warps per SM), two rows per thread 860 (five
// warps), and 624 the kernel that evaluated nodes one by one, lane = row.  Depth 5: 280, depth 7:
// 1170 (1940 with node-by-node decisions), depth 8: 2560 (6350; slots in twelve floats, three
// loads per gather).
//
// The kernels are templates of the depth; every depth is instantiated in its own
// translation unit so that they compile in parallel.
#pragma once
#include <algorithm>

#include "tree_layout.h"
#include "launch.h"
#include "wdf_device.cuh"

namespace wdf {

// Warps per SM that the registers allow: at depth 6, 20 (96 registers) measured no faster than
// 16 and 12 (168) 5 % slower.
constexpr int kExplainWarps = 16;

// Depth 8 leaves the L1 cache a good part of the SM's memory: a gather in flight holds its lines
// there, some 300 KB for twelve warps if they could, and waits for them otherwise.  233,472 rows and
// 40 trees of 134 features with blocks in up to 132 / 164 / 196 / 228 KB: 2773 / 2655 / 2869 / 2865 us;
// 191 features (four blocks in 164 KB) are as fast in all of it, 60 features (ten) 2 % faster by
// the driver's choice; depth 5 to 7 do not gain.
constexpr size_t kExplainCarveout = (size_t)164 << 10;
constexpr bool explain_carveout(int D, int tile_rows, size_t smem) {
    const size_t blocks = kExplainCarveout / (smem + 1024);
    return D == 8 && tile_rows == 32 && blocks >= 5 && blocks <= 8;
}

template <int D>
struct ExplainCfg {
    static constexpr int TOP = unit_top(D), UPT = units_per_tree(D);  // levels above the units, units
    static constexpr int GS = gather_group(D);                        // bottom subtrees of a unit
    static constexpr int LW = lines_words(D);
    // deep trees loop over their units (unrolled, the code of a tree does not stay in the
    // instruction cache)
    static constexpr int UNROLL = D >= 7 ? 1 : UPT;
};
WDF_HD constexpr int explain_threads(int tc) { return 2 * tc; }

// Shared memory of one block: code tile (TC / 32 blocks of quads) | phi tile ((F + 1) x (TC + 1)
// floats, feature-major, row F a scratch row; wide: no code tile and rows of TC floats) | per warp, a ring of SLOTS chunks and their line
// maps, then the nodes above a tree's units.  (Depth 8 a tree at a time, 33.5 KB a block instead
// of 24.7: 3063 us where the above took 2655, 3371 where 191 features take 3090; depth 7 a unit
// at a time 3 % slower.)
template <int D>
struct ExLayout {
    size_t x, p, total;
    // a chunk is copied while the one (of two units) or the two before it are processed
    static constexpr int SLOTS = chunk_units(D) > 1 ? 2 : 3;
    static constexpr int LINE = chunk_bytes(D), SLOT = LINE + (chunk_units(D) > 2 ? 8 * chunk_units(D) : 16);
    static constexpr int WARP = SLOTS * SLOT + (unit_top(D) > 1 ? 8 * (int)sizeof(UnitNode) : 0);
    __host__ __device__ ExLayout(int F, int quads, int TC, bool wide = false) {
        x = wide ? 0 : (size_t)(TC / 32) * quads * 16;
        p = ((size_t)(F + 1) * (wide ? TC : TC + 1) * 4 + 15) & ~(size_t)15;
        total = x + p + (size_t)(TC / 16) * WARP;
    }
};

// 16-byte and 32-byte read-only loads predicated on `on` (the outputs keep their values
// when off): a dead bottom subtree issues no load.  Without a line of their own in the L1 cache
// (one gather in four hits it at depth 6, one in twenty-five at depth 8) the gathers in flight
// wait less for one: 233,472 rows, depth 5 to 8 1391 -> 1349, 1409 -> 1358, 2321 -> 2202, 2637 -> 2580 us
// (200, 100, 80, 40 trees).  (A branch around the loads makes the
// compiler wait for them at its end, and sending a dead subtree's rows to one entry costs the
// eight wavefronts that return 32 bytes to 32 lanes.)
__device__ __forceinline__ void ldg_f4_if(const void *p, float4 &r, uint32_t on) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.u32 q, %5, 0;\n@q ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];\n}\n"
        : "+f"(r.x), "+f"(r.y), "+f"(r.z), "+f"(r.w)
        : "l"(p), "r"(on));
}

// One 32-byte vector in a single 256-bit load (the address is 32-byte aligned).
__device__ __forceinline__ void ldg_f8_if(const void *p, float4 &a, float4 &b, uint32_t on) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.u32 q, %9, 0;\n@q ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n}\n"
        : "+f"(a.x), "+f"(a.y), "+f"(a.z), "+f"(a.w), "+f"(b.x), "+f"(b.y), "+f"(b.z), "+f"(b.w)
        : "l"(p), "r"(on));
}

// phi[o[q]] += val[q] for the first cnt positions of a batch that repeats features: first the
// positions of a feature's first occurrence, then (rep) the others, which are distinct among
// themselves, or (rep 0xFF) all one after another.  Kept out of line so the per-tree loop
// stays small in the instruction cache.
static __device__ __noinline__ void flush_repeats(float *myphi, int4 oa, int4 ob, float4 va, float4 vb, int cnt,
                                                  uint32_t rep) {
    const int o[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
    const float v[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
    if (rep == 0xFFu) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < cnt) myphi[o[q]] += v[q];
        return;
    }
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        float a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < cnt && (int)((rep >> q) & 1u) == pass) a[q] = myphi[o[q]];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < cnt && (int)((rep >> q) & 1u) == pass) myphi[o[q]] = a[q] + v[q];
    }
}

// phi[o[q]] += val[q] for the first cnt positions of one flush batch.  fast: the batch
// repeats no real feature, so all reads may precede all writes.  Pass-through positions
// (the scratch row) are not skipped: a predicated-off shared access still takes an L1
// data-pipe wavefront (ncu), so a test per position only added instructions.
__device__ __forceinline__ void flush_batch(float *myphi, const int (&o)[8], const float (&val)[8], int cnt, bool fast,
                                            const unsigned char *rep) {
    if (fast) {
        float a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < cnt) a[q] = myphi[o[q]];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < cnt) myphi[o[q]] = a[q] + val[q];
    } else {
        flush_repeats(myphi, make_int4(o[0], o[1], o[2], o[3]), make_int4(o[4], o[5], o[6], o[7]),
                      make_float4(val[0], val[1], val[2], val[3]), make_float4(val[4], val[5], val[6], val[7]), cnt,
                      *rep);
    }
}

__device__ __forceinline__ void load_offsets8(const uint16_t *p, int (&o)[8]) {
    const uint4 a = *reinterpret_cast<const uint4 *>(p);
    o[0] = (int)(a.x & 0xFFFFu); o[1] = (int)(a.x >> 16); o[2] = (int)(a.y & 0xFFFFu); o[3] = (int)(a.y >> 16);
    o[4] = (int)(a.z & 0xFFFFu); o[5] = (int)(a.z >> 16); o[6] = (int)(a.w & 0xFFFFu); o[7] = (int)(a.w >> 16);
}

// The gathered entries of a unit's bottom subtrees: Q float4 each and, at depth 8, the root's
// slot apart.
template <int D>
struct UnitSlots {
    static constexpr int GS = gather_group(D), Q = slots_per_entry(D) / 4;
    float4 v[GS][Q];
    float x0[GS];
    // slot k of subtree j (both compile-time constants after unrolling)
    __device__ __forceinline__ float slot(int j, int k) const {
        if (extra_slots(D) && k == 0) return x0[j];
        const int at = k - extra_slots(D);
        const float4 &x = v[j][at >> 2];
        return (at & 3) == 0 ? x.x : (at & 3) == 1 ? x.y : (at & 3) == 2 ? x.z : x.w;
    }
};

// Entries and gathers of unit u of tree t: live and lm are the live flags and line maps of its
// subtrees, w and topw the row's decisions in the unit and at the nodes above the units.
template <int D>
__device__ __forceinline__ void gather_unit(const float *sfold, int T, int t, int u, uint32_t live,
                                            const uint32_t (&lm)[(gather_group(D) + 3) / 4], uint32_t w, uint32_t topw,
                                            UnitSlots<D> &v) {
    using S = Shape<D>;
    constexpr int GS = UnitSlots<D>::GS, Q = UnitSlots<D>::Q, TOP = unit_top(D);
    constexpr uint32_t EB = 4 * S::SP;  // bytes of an entry
    // decisions on the path to the unit's root, then R of the children of every node above its
    // bottom subtrees (wdf_internal.h), in units of 8 entries repeated twice (line_pos), in bytes
    constexpr uint32_t ONE = EB * ((1u << (D + 1)) + 1u);
    uint32_t path = 0u, R[GS > 1 ? GS - 1 : 1];
#pragma unroll
    for (int k = 0; k < TOP; ++k) path = (path << 1) | ((topw >> ((1 << k) - 1 + (u >> (TOP - k)))) & 1u);
    R[0] = 0u;
#pragma unroll
    for (int k = 0; k < GS - 1; ++k)
        R[k] = 2u * (k == 0 ? path * (8u * ONE) : R[(k - 1) >> 1]) + ((w >> k) & 1u) * (8u * ONE);
    const char *tf = reinterpret_cast<const char *>(sfold) + ((size_t)t * S::NS + u * GS) * S::E * EB;
    const char *tx =
        reinterpret_cast<const char *>(sfold + (size_t)T * S::NS * S::E * S::SP + ((size_t)t * S::NS + u * GS) * S::E);
#pragma unroll
    for (int j = 0; j < GS; ++j) {
        const uint32_t on = (live >> j) & 1u;
        const uint32_t e = (GS > 1 ? R[(GS - 2 + j) >> 1] : 0u) + ((w >> (GS - 1 + 3 * j)) & 7u) * ONE;
        // the shift amount is the low five bits of the map's byte
        const uint32_t at = __funnelshift_r(e, 0u, lm[j >> 2] >> (8 * (j & 3))) & ((S::E - 1) * EB);
#pragma unroll
        for (int k = 0; k < Q; ++k) v.v[j][k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if constexpr (Q == 2) ldg_f8_if(tf + j * (int)(S::E * EB) + at, v.v[j][0], v.v[j][Q - 1], on);
        else ldg_f4_if(tf + j * (int)(S::E * EB) + at, v.v[j][0], on);
        if (extra_slots(D))
            asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v.x0[j]) : "l"(tx + j * (int)(S::E * 4) + at / 8));
        else
            v.x0[j] = 0.0f;
    }
}

// Values of the nodes above a unit's bottom subtrees: up, inside the unit (heap order); top, the
// nodes above the units, on the unit's path (the first unit below one starts its sum).
template <int D>
__device__ __forceinline__ void unit_sums(const UnitSlots<D> &v, int u, float (&up)[gather_group(D) > 1 ? gather_group(D) - 1 : 1],
                                          float (&top)[units_per_tree(D) > 1 ? units_per_tree(D) - 1 : 1]) {
    constexpr int GS = gather_group(D), TOP = unit_top(D), LG = ilog2(GS);
#pragma unroll
    for (int k = 0; k < GS - 1; ++k) up[k] = 0.0f;
#pragma unroll
    for (int j = 0; j < GS; ++j)
#pragma unroll
        for (int l = 0; l < LG; ++l) up[(1 << l) - 1 + (j >> (LG - l))] += v.slot(j, TOP + l);
#pragma unroll
    for (int k = 0; k < TOP; ++k) {
        float x = v.slot(0, k);
#pragma unroll
        for (int j = 1; j < GS; ++j) x += v.slot(j, k);
        const int node = u >> (TOP - k);
#pragma unroll
        for (int p = 0; p < 1 << k; ++p) {
            float &tp = top[(1 << k) - 1 + p];
            if (p == node) tp = u & ((1 << (TOP - k)) - 1) ? tp + x : x;
        }
    }
}

// One tile of TC consumer rows starting at row c0 (of n rows), for one ensemble: parts
// [part0, part1) of its trees.  With scratch null the parts are all of them, the first stored
// into phi, the others added; else part p is stored at scratch + p * n * F, row stride F, and
// k_add_parts adds them.  The rows' decision codes are copied from codes, the code blocks of all n rows written by k_encode_slices or
// k_encode_batch (padded to a multiple of TC rows).
//
// Two warps share 32 rows, their codes and their phi columns: the first takes the even trees of
// a part, the second the odd ones, and they take turns -- while one adds a unit's values into
// phi, the other makes its next decisions and has its next gathers in flight.  A row's phi
// fixes how many rows an SM can hold; two warps per 32 rows double the warps that hide the
// gathers' and the shared memory's latency.  The turns also fix the order of the additions.
//
// WIDE: the form of ensembles whose tile does not fit a block's shared memory otherwise (from some
// 1,400 features of 16 to 255 thresholds on, to about 1,770).  The codes are read where they lie, in global memory, and a
// feature's phi row is 32 floats, rotated by the feature's number (row r of feature f in word (r + f)
// mod 32) so that its storing reads all banks, as the 33 floats of the other form do.  The same
// additions in the same order.  48,640 rows, 17 thresholds a feature, on both sides of the border (the
// other form / this one): depth 6 18.0 / 18.6 ms (380 trees, 1,390 / 1,405 features), depth 7 15.9 / 20.1
// (185, 1,375 / 1,402), depth 8 16.9 / 14.8 (94, 1,375 / 1,400); so the other form stays where it fits.
template <int D, int TC, bool WIDE>
__device__ __forceinline__ void explain_tile(const ExplainJob &job, const unsigned char *__restrict__ codes,
                                             int64_t n, float *__restrict__ phi, int64_t ldp, int64_t c0, int part0,
                                             int part1, float *__restrict__ scratch, unsigned char *smem_raw) {
    using X = ExplainCfg<D>;
    static_assert(!WIDE || TC == 32, "wide tiles have 32 rows");
    constexpr int XS = WIDE ? TC : TC + 1, GS = X::GS, TOP = X::TOP, UPT = X::UPT;
    constexpr int NT = explain_threads(TC), SLOTS = ExLayout<D>::SLOTS, SLOT = ExLayout<D>::SLOT;
    constexpr int FB = flush_group_bottom(D), GL = flush_group_len(D), LW = X::LW;
    constexpr int IMG = image_bytes(D), CHUNK = chunk_bytes(D), LINE = ExLayout<D>::LINE;
    constexpr int CU = chunk_units(D), CPT = tree_chunks(D);
    const int F = job.F, T = job.T, quads = job.sa.quads;
    const ExLayout<D> L(F, quads, TC, WIDE);
    uint4 *sx = reinterpret_cast<uint4 *>(smem_raw);
    float *sp = reinterpret_cast<float *>(smem_raw + L.x);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, pair = warp >> 1, half = warp & 1;
    unsigned char *ring = smem_raw + L.x + L.p + (size_t)warp * ExLayout<D>::WARP;  // this warp's
    const uint2 *above = reinterpret_cast<const uint2 *>(ring + SLOTS * SLOT);
    const uint4 *src = reinterpret_cast<const uint4 *>(codes) + (c0 / 32) * quads;
    if (!WIDE)
        for (int i = tid; i < TC / 32 * quads; i += NT) sx[i] = __ldg(src + i);
    for (int i = tid; i < (F + 1) * XS; i += NT) sp[i] = 0.0f;
    float *myphi = WIDE ? sp : sp + 32 * pair + lane;
    const uint4 *block = WIDE ? src : sx + pair * quads;
    // this lane's phi in the row that starts at o (a multiple of 32 x feature)
    auto rotate = [&](int (&o)[8]) {
        if (WIDE) {
#pragma unroll
            for (int q = 0; q < 8; ++q) o[q] += (lane + (o[q] >> 5)) & 31;
        }
    };
    auto turn = [&]() {
        // constant barrier numbers: a block with a variable one reserves all sixteen, and an SM
        // holds four such blocks
        if (TC == 32 || pair == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
        else if (TC == 64 || pair == 1) asm volatile("bar.sync 2, 64;" ::: "memory");
        else if (pair == 2) asm volatile("bar.sync 3, 64;" ::: "memory");
        else asm volatile("bar.sync 4, 64;" ::: "memory");
    };

    // Copies chunk c of tree t into a slot of the ring, with a tree's first chunk the nodes above
    // its units too (read with the decisions of its first unit, CPT chunks before the next copy).
    const unsigned char *image = job.image + (size_t)(ilog2(TC) - 5) * T * IMG;
    auto stage = [&](int t, int c, const unsigned char *slot) {
        const unsigned char *tree = image + (size_t)t * IMG;
#pragma unroll
        for (int i = 0; i < CHUNK / 16 + (TOP > 1 ? 4 : 0); i += 32) {
            const unsigned char *src = tree + c * CHUNK + 16 * (i + lane);
            uint32_t dst = (uint32_t)__cvta_generic_to_shared(slot) + 16 * (i + lane);
            bool on = i + lane < CHUNK / 16;
            if (TOP > 1 && c == 0 && i + 32 >= CHUNK / 16 + 4 && lane >= 28) {
                src = tree + image_top(D) + 16 * (lane - 28);
                dst = (uint32_t)__cvta_generic_to_shared(above) + 16 * (lane - 28);
                on = true;
            }
            if (on) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
        }
        // the line maps: two words a unit (a tree has at least four)
        const uint32_t ldst = (uint32_t)__cvta_generic_to_shared(slot) + LINE;
        const uint32_t *lsrc = job.lines + (size_t)t * LW + c * CU * (GS / 4);
        if (CU == 1) {
            if (lane == 24) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ldst), "l"(lsrc) : "memory");
        } else if (lane < CU / 2) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ldst + 16 * lane), "l"(lsrc + 4 * lane) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto arrived = [&]() {  // all copies but the newest SLOTS - 2 groups are in shared memory
        asm volatile("cp.async.wait_group %0;" ::"n"(SLOTS - 2) : "memory");
        __syncwarp();
    };

    // Decisions of one unit for this lane's row, and of its tree's nodes above the units (bit =
    // node).
    struct Words {
        uint32_t w, top;
    };
    auto decide = [&](const unsigned char *slot, int u, int i, const Words &p) -> Words {
        Words q = p;
        const uint2 *rec = reinterpret_cast<const uint2 *>(slot) + i * 32;
        if (TOP > 1 && u == 0) {
            uint32_t w[2] = {unit_decide(rec[lane], block, job.sa),
                             lane < UPT - 1 ? unit_decide(above[lane], block, job.sa) : 0u};
            transpose32(w, lane);
            q.w = w[0];
            q.top = w[1];
        } else {
            q.w = transpose32(unit_decide(rec[lane], block, job.sa), lane);
            if (TOP == 1 && u == 0) q.top = q.w >> 31;
        }
        return q;
    };
    UnitSlots<D> v;
    auto gather = [&](int t, const unsigned char *slot, int u, int i, const Words &p, bool mine) {
        const uint32_t live = reinterpret_cast<const uint32_t *>(slot + chunk_flags(D))[i];
        uint32_t lm[(GS + 3) / 4];
#pragma unroll
        for (int k = 0; k < (GS + 3) / 4; ++k)
            lm[k] = reinterpret_cast<const uint32_t *>(slot + LINE)[i * (GS / 4) + k];
        gather_unit<D>(job.sfold, T, t, u, mine ? live : 0u, lm, p.w, p.top, v);
    };
    float top[UPT > 1 ? UPT - 1 : 1];
    // Adds unit u's node values into phi; the top nodes' sums are kept until the tree's last unit.
    auto flush = [&](const unsigned char *slot, int u, int i, bool mine) {
        const uint16_t *off = reinterpret_cast<const uint16_t *>(slot + chunk_offsets(D)) + i * GL;
        const uint32_t flags = reinterpret_cast<const uint32_t *>(slot + chunk_flags(D))[i];
        const uint32_t fok = flags >> 8, real = (flags >> 16) & (mine ? ~0u : 0u);
        const unsigned char *rep = slot + chunk_repeats(D) + i * (GL / 8);
        int o[8];
        load_offsets8(off, o);
        rotate(o);
        float up[GS > 1 ? GS - 1 : 1];
        unit_sums<D>(v, u, up, top);
#pragma unroll
        for (int b = 0; b < GL / 8; ++b) {
            int on[8];
            if (b + 1 < GL / 8) {  // off the chain of phi round trips
                load_offsets8(off + 8 * (b + 1), on);
                rotate(on);
            }
            float x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (b < FB / 8)  // two subtrees to a batch
                    x[q] = q < 6 ? v.slot(2 * b + q / 3 < GS ? 2 * b + q / 3 : 0, D - 2 + q % 3) : 0.0f;
                else
                    x[q] = q < GS - 1 ? up[q < GS - 1 ? q : 0] : 0.0f;
            }
            if ((real >> b) & 1u)
                flush_batch(myphi, o, x, b < FB / 8 ? (GS > 1 ? 6 : 3) : GS - 1, (fok >> b) & 1u, rep + b);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (b + 1 < GL / 8) o[q] = on[q];
        }
        if (UPT > 1 && u == UPT - 1 && mine) {
            load_offsets8(off + (CU - i) * GL, o);
            rotate(o);
            float x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = q < UPT - 1 ? top[q < UPT - 1 ? q : 0] : 0.0f;
            flush_batch(myphi, o, x, UPT - 1, (fok >> (GL / 8)) & 1u, rep + (CU - i) * (GL / 8));
        }
    };

    const int P = explain_parts(T, D);
    __syncthreads();  // the code tile and the zeroed phi tile
    for (int part = part0; part < part1; ++part) {
        const int tb = (int)((long long)T * part / P), te = (int)((long long)T * (part + 1) / P);
        // both warps take the same number of turns; past the part's end the second repeats a tree
        // without gathers and additions (a branch around the gathers would wait for them)
        auto tree = [&](int t) { return min(t, te - 1); };
        // chunk c + k of tree t, past the tree's end of the warp's next trees
        auto stage_ahead = [&](int t, int c, int k, const unsigned char *slot) {
            stage(tree(t + 2 * ((c + k) / CPT)), (c + k) % CPT, slot);
        };
        // the chunk at work, the next one and (of three) the one to copy into
        const unsigned char *now = ring, *next = ring + SLOT, *free = ring + (SLOTS - 1) * SLOT;
        stage_ahead(tb + half, 0, 0, now);
        if (SLOTS == 3) stage_ahead(tb + half, 0, 1, next);
        arrived();
        Words p = decide(now, 0, 0, Words{});
        if (half) turn();
        for (int t = tb + half; t < te + half; t += 2) {
            const bool mine = t < te;
#pragma unroll 1
            for (int c = 0; c < CPT; ++c) {
                stage_ahead(t, c, SLOTS - 1, free);
#pragma unroll X::UNROLL
                for (int i = 0; i < CU; ++i) {
                    const int u = c * CU + i;
                    const bool last = i + 1 == CU;
                    gather(tree(t), now, u, i, p, mine);
                    if (last) arrived();
                    p = decide(last ? next : now, u + 1 < UPT ? u + 1 : 0, last ? 0 : i + 1, p);
                    turn();
                    flush(now, u, i, mine);
                    turn();
                }
                const unsigned char *done = now;
                now = next;
                next = SLOTS == 3 ? free : done;
                free = done;
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");  // copies past the end: their slots are staged anew
        if (!half) turn();
        // the part's sums, stored or added, and the tile zeroed for the next part
        for (int r = half; r < 32; r += 2) {
            const int64_t row = c0 + 32 * pair + r;
            if (row >= n) break;
            float *dst = scratch ? scratch + ((size_t)part * n + row) * F : phi + row * ldp;
            for (int f = lane; f < F; f += 32) {
                float &y = sp[f * XS + (WIDE ? (r + f) & 31 : 32 * pair + r)];
                const float x = y;
                dst[f] = part > part0 && !scratch ? dst[f] + x : x;
                y = 0.0f;
            }
        }
        turn();
    }
}

// Block (tile, y): parts [P y / gridDim.y, P (y + 1) / gridDim.y) of the tile's rows (scratch
// non-null when there is more than one y).
template <int D, int TC, bool WIDE>
__global__ void __launch_bounds__(explain_threads(TC), WIDE ? 1 : kExplainWarps * 16 / TC) k_explain(const unsigned char *__restrict__ codes, int64_t n, ExplainJob job, float *__restrict__ phi, int64_t ldp,
              float *__restrict__ scratch) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = explain_parts(job.T, D), y = blockIdx.y, Y = gridDim.y;
    explain_tile<D, TC, WIDE>(job, codes, n, phi, ldp, (int64_t)blockIdx.x * TC, P * y / Y, P * (y + 1) / Y, scratch, smem_raw);
}

// Few rows: the node values of 32 rows and one tree per warp, every tree at once, position i of
// the flush order at values + (((row block) * T + t) * flush_len + i) * 32 + row;
// k_sum_values then adds each feature's in the order of the tile kernel.  Latency-bound.
constexpr int kValueWarps = 4;
template <int D>
__global__ void __launch_bounds__(32 * kValueWarps) k_values(const unsigned char *__restrict__ codes, ExplainJob job,
                                                            float *__restrict__ values) {
    using X = ExplainCfg<D>;
    constexpr int GS = X::GS, TOP = X::TOP, UPT = X::UPT, LW = X::LW;
    constexpr int FB = flush_group_bottom(D), GL = flush_group_len(D), FL = flush_len(D);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, quads = job.sa.quads;
    uint4 *block = reinterpret_cast<uint4 *>(smem_raw);
    const int t = blockIdx.x * kValueWarps + (tid >> 5), tt = min(t, job.T - 1);
    const uint2 *rec = reinterpret_cast<const uint2 *>(job.sa.unit) + (size_t)tt * UPT * 32;
    const unsigned char *chunk = job.image + (size_t)tt * image_bytes(D) + lane / chunk_units(D) * chunk_bytes(D);
    const uint32_t flags =
        lane < UPT ? __ldg(reinterpret_cast<const uint32_t *>(chunk + chunk_flags(D)) + lane % chunk_units(D)) : 0u;
    const uint4 *src = reinterpret_cast<const uint4 *>(codes) + (size_t)blockIdx.y * quads;
    uint2 node = __ldg(rec + lane);
    early_launch();
    previous_done();  // the rows' codes
    for (int i = tid; i < quads; i += 32 * kValueWarps) block[i] = src[i];
    __syncthreads();
    if (t >= job.T) return;
    uint32_t topw = 0u;
    if (TOP > 1)
        topw = transpose32(lane < UPT - 1 ? unit_decide(__ldg(rec + lane * 32 + 31), block, job.sa) : 0u, lane);
    float *out = values + ((size_t)blockIdx.y * job.T + t) * FL * 32 + lane;
    float top[UPT > 1 ? UPT - 1 : 1];
#pragma unroll X::UNROLL
    for (int u = 0; u < UPT; ++u) {
        const uint32_t w = transpose32(unit_decide(node, block, job.sa), lane);
        if (TOP == 1 && u == 0) topw = w >> 31;
        uint32_t lm[(GS + 3) / 4];
#pragma unroll
        for (int k = 0; k < (GS + 3) / 4; ++k) lm[k] = __ldg(job.lines + (size_t)t * LW + u * (GS / 4) + k);
        UnitSlots<D> v;
        const uint32_t unit_flags = __shfl_sync(0xFFFFFFFFu, flags, u);
        gather_unit<D>(job.sfold, job.T, t, u, unit_flags, lm, w, topw, v);
        if (u + 1 < UPT) node = __ldg(rec + (u + 1) * 32 + lane);
        float up[GS > 1 ? GS - 1 : 1];
        unit_sums<D>(v, u, up, top);
        const uint32_t some = unit_flags >> 16;
        float *dst = out + (size_t)u * GL * 32;
#pragma unroll
        for (int b = 0; b < GL / 8; ++b) {
            if (!((some >> b) & 1u)) continue;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (b < FB / 8) {
                    if (q < 6 && 2 * b + q / 3 < GS)
                        dst[(8 * b + q) * 32] = v.slot(2 * b + q / 3 < GS ? 2 * b + q / 3 : 0, D - 2 + q % 3);
                } else if (q < GS - 1) {
                    dst[(8 * b + q) * 32] = up[q < GS - 1 ? q : 0];
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < UPT - 1; ++k) out[(size_t)(UPT * GL + k) * 32] = top[k];
}

// Persistent form over a ragged batch: work item i is a tile of a request, or one of its groups
// of parts (launch.h).  Blocks claim items in order from a counter (n_items[1], zero at launch),
// so expensive items, which the host puts first, spread over the whole grid and cheap ones fill
// the tail.  The item count n_items[0] is read from device memory, so one captured graph serves
// batches of any size up to its capacity.  Which block computes a tile does not change any
// row's arithmetic, nor do the groups: parts are always added in their order.
template <int D, int TC, bool WIDE>
__global__ void __launch_bounds__(explain_threads(TC), WIDE ? 1 : kExplainWarps * 16 / TC) k_explain_batch(const ExplainJob *__restrict__ jobs,
                                                         const BatchRequest *__restrict__ reqs,
                                                         const int4 *__restrict__ items, int *n_items) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int claimed, arrived;
    const int count = n_items[0];
    for (;;) {
        if (threadIdx.x == 0) claimed = atomicAdd(n_items + 1, 1);
        __syncthreads();
        const int i = claimed;
        if (i >= count) break;
        const int4 it = items[i];
        const ExplainJob job = jobs[it.x];
        const BatchRequest rq = reqs[it.y];
        const int group = it.z >> kBatchGroupShift, P = explain_parts(job.T, D), groups = rq.groups;
        const int64_t c0 = ((int64_t)(it.z & ((1 << kBatchGroupShift) - 1)) << 31) | (uint32_t)it.w;
        explain_tile<D, TC, WIDE>(job, rq.codes, rq.n, rq.phi, rq.ldp, c0, P * group / groups, P * (group + 1) / groups,
                            groups > 1 ? rq.parts : nullptr, smem_raw);
        __syncthreads();
        if (groups > 1) {  // the last of the tile's items adds its parts
            if (threadIdx.x == 0) {
                __threadfence();
                arrived = atomicAdd(n_items + 2 + rq.tile0 + (int)(c0 / TC), 1);
                __threadfence();
            }
            __syncthreads();
            if (arrived == groups - 1) {
                const int64_t rows = min((int64_t)TC, rq.n - c0), cells = rows * job.F, step = rq.n * job.F;
                const float *src = rq.parts + c0 * job.F;
                for (int64_t k = threadIdx.x; k < cells; k += explain_threads(TC)) {
                    float x = __ldcg(src + k);
                    for (int p = 1; p < P; ++p) x += __ldcg(src + p * step + k);
                    rq.phi[(c0 + k / job.F) * rq.ldp + k % job.F] = x;
                }
            }
            __syncthreads();
        }
    }
}

// The part of an SM's memory that a kernel's blocks want (228 KB in all).
template <class K>
cudaError_t set_carveout(K kern, int D, int tile_rows, size_t smem) {
    const int percent = explain_carveout(D, tile_rows, smem) ? (int)(100 * (kExplainCarveout >> 10) / 228 + 1)
                                                             : cudaSharedmemCarveoutDefault;
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, percent);
}

template <int D, int TC, bool WIDE>
cudaError_t explain_t(const unsigned char *codes, int64_t n, const ExplainJob &job, float *phi, int64_t ldp,
                      int splits, float *scratch, const DevInfo &dev, cudaStream_t st) {
    const size_t smem = ExLayout<D>(job.F, job.sa.quads, TC, WIDE).total;
    auto kern = k_explain<D, TC, WIDE>;
    cudaError_t err = allow_shared(kern, smem, dev);
    if (err == cudaSuccess) err = set_carveout(kern, D, TC, smem);
    if (err != cudaSuccess) return err;
    const int64_t blocks = (n + TC - 1) / TC;
    kern<<<dim3((unsigned)blocks, (unsigned)splits), explain_threads(TC), smem, st>>>(codes, n, job, phi, ldp, scratch);
    count_launches(1);
    return cudaGetLastError();
}

template <int D>
cudaError_t values_t(const unsigned char *codes, int64_t n, const ExplainJob &job, float *values, const DevInfo &dev,
                     cudaStream_t st) {
    const size_t smem = (size_t)job.sa.quads * 16;
    auto kern = k_values<D>;
    cudaError_t err = allow_shared(kern, smem, dev);
    if (err != cudaSuccess) return err;
    const dim3 grid((unsigned)((job.T + kValueWarps - 1) / kValueWarps), (unsigned)((n + 31) / 32));
    err = launch_dependent(kern, grid, 32 * kValueWarps, smem, st, codes, job, values);
    count_launches(1);
    return err != cudaSuccess ? err : cudaGetLastError();
}

template <int D, int TC, bool WIDE>
cudaError_t batch_t(const ExplainJob *jobs, const BatchRequest *reqs, const int4 *items, int *n_items, int F_max,
                    int q_max, int grid, const DevInfo &dev, cudaStream_t st) {
    const size_t smem = ExLayout<D>(F_max, q_max, TC, WIDE).total;
    auto kern = k_explain_batch<D, TC, WIDE>;
    cudaError_t err = allow_shared(kern, smem, dev, kBatchShared);
    if (err == cudaSuccess) err = set_carveout(kern, D, TC, smem);
    if (err != cudaSuccess) return err;
    if (grid <= 0) grid = dev.sms * explain_blocks_per_sm(D, F_max, q_max, TC, dev);
    kern<<<grid, explain_threads(TC), smem, st>>>(jobs, reqs, items, n_items);
    count_launches(1);
    return cudaGetLastError();
}

// Explicit instantiation of the kernels of one (depth, tile rows) pair; each pair is
// compiled in one of the k_explain_d*.cu translation units.
#define WDF_EXPLAIN_FORM(d, tc, wide, spec)                                                                      \
    spec template cudaError_t explain_t<d, tc, wide>(const unsigned char *, int64_t, const ExplainJob &, float *, \
                                                     int64_t, int, float *, const DevInfo &, cudaStream_t);      \
    spec template cudaError_t batch_t<d, tc, wide>(const ExplainJob *, const BatchRequest *, const int4 *, int *, \
                                                   int, int, int, const DevInfo &, cudaStream_t);
#define WDF_EXPLAIN_TILE(d, tc, spec) WDF_EXPLAIN_FORM(d, tc, false, spec)
#define WDF_EXPLAIN_WIDE(d, spec) WDF_EXPLAIN_FORM(d, 32, true, spec)
#define WDF_EXPLAIN_VALUES(d, spec)                                                                              \
    spec template cudaError_t values_t<d>(const unsigned char *, int64_t, const ExplainJob &, float *,           \
                                          const DevInfo &, cudaStream_t);
#define WDF_EXPLAIN_DEPTH(d, spec) WDF_EXPLAIN_TILE(d, 32, spec) WDF_EXPLAIN_TILE(d, 64, spec) \
    WDF_EXPLAIN_TILE(d, 128, spec) WDF_EXPLAIN_VALUES(d, spec)

}  // namespace wdf
