// Device helpers shared by the kernels: tree shapes, decisions on sliced codes
// (tree_layout.h), entries of the bottom subtrees.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "launch.h"
#include "tree_layout.h"

namespace wdf {

template <int D>
struct Shape {
    static constexpr int NI = (1 << D) - 1;    // inner nodes
    static constexpr int NL = 1 << D;          // leaves
    static constexpr int NS = 1 << (D - 2);    // bottom subtrees
    static constexpr int E = 1 << (D + 1);     // entries per bottom subtree
    static constexpr int NW = (NI + 31) / 32;  // 32-bit decision words
    static constexpr int SP = slots_per_entry(D);  // slots of an entry's vector
};

__device__ __forceinline__ TreeMeta load_meta(const TreeMeta *p) {
    TreeMeta m;
    const uint2 *src = reinterpret_cast<const uint2 *>(p);
    uint2 *dst = reinterpret_cast<uint2 *>(&m);
#pragma unroll
    for (int i = 0; i < (int)(sizeof(TreeMeta) / sizeof(uint2)); ++i) dst[i] = __ldg(src + i);
    return m;
}

template <int D>
__device__ __forceinline__ uint32_t dbit(const uint32_t (&dw)[Shape<D>::NW], int v) {
    return (dw[v >> 5] >> (v & 31)) & 1u;
}

// Two adjacent decision bits, v and v + 1 (bit 0 = node v), of the decision words.
template <int D>
__device__ __forceinline__ uint32_t dbit2(const uint32_t (&dw)[Shape<D>::NW], int v) {
    if ((v & 31) != 31) return (dw[v >> 5] >> (v & 31)) & 3u;
    return ((dw[v >> 5] >> 31) | (dw[(v >> 5) + 1] << 1)) & 3u;
}

// Entry index of the row at every bottom subtree (wdf_internal.h): the ancestors' raw
// decisions R are built once per node of depth < D-2 (siblings share them), then each
// entry takes d_r and the adjacent pair d_{2r+1}, d_{2r+2} in one extraction.
template <int D>
__device__ __forceinline__ void subtree_entries(const uint32_t (&dw)[Shape<D>::NW], uint32_t (&ent)[Shape<D>::NS]) {
    constexpr int NS = Shape<D>::NS;
    uint32_t R[NS > 1 ? NS - 1 : 1];  // R of the children of node v, v < NS - 1
#pragma unroll
    for (int v = 0; v < NS - 1; ++v) R[v] = ((v == 0 ? 0u : R[(v - 1) >> 1]) << 1) | dbit<D>(dw, v);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const int r = NS - 1 + s;
        const uint32_t Rr = r == 0 ? 0u : R[(r - 1) >> 1];
        ent[s] = (Rr << 3) | (dbit<D>(dw, r) << 2) | dbit2<D>(dw, 2 * r + 1);
    }
}

// Lets blocks of a kernel take smem bytes of dynamic shared memory beside `fixed` of its own.  The
// limit belongs to the kernel, not to the launch, so every caller sets the same one, all that
// a block may have: with each call's own size, host threads in calls on different ensembles
// lowered it under one another between setting it and launching.
template <class K>
inline cudaError_t allow_shared(K kern, size_t smem, const DevInfo &dev, size_t fixed = 0) {
    if (smem + fixed > dev.smem_optin) return cudaErrorInvalidConfiguration;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(dev.smem_optin - fixed));
}

// Dependent launches (launch_dependent): early lets the next kernel's blocks start once all blocks
// of this one are under way; previous_done waits for the kernel before, whose results the
// next loads may read.
__device__ __forceinline__ void early_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void previous_done() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launches a kernel that starts while the one before it on st ends: it may read that one's
// results, and write what earlier ones read, only after previous_done().  (A call of few rows
// is three short kernels; one row and 100 trees of depth 6 72 -> 60 us alone, 30.7 -> 29.1 back to
// back; 777 rows and 500 trees of depth 7 128.8 -> 126.4.)
template <class... A>
inline cudaError_t launch_dependent(void (*kern)(A...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st,
                                    A... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Transposes of N 32 x 32 bit matrices whose row r is lane r's word: lane b gets bit b of
// every lane's word, in lane order.  The matrices' exchanges are interleaved.
template <int N>
__device__ __forceinline__ void transpose32(uint32_t (&w)[N], int lane) {
    uint32_t y[N];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const bool up = lane & s;
#pragma unroll
        for (int i = 0; i < N; ++i) y[i] = __shfl_xor_sync(0xFFFFFFFFu, w[i], s);
        if (s >= 8) {  // whole bytes
            const uint32_t sel = s == 16 ? (up ? 0x3276u : 0x5410u) : (up ? 0x3715u : 0x6240u);
#pragma unroll
            for (int i = 0; i < N; ++i) w[i] = __byte_perm(w[i], y[i], sel);
        } else {
            const uint32_t low = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
            const uint32_t keep = up ? ~low : low;
#pragma unroll
            for (int i = 0; i < N; ++i)
                w[i] = (w[i] & keep) | (__funnelshift_l(y[i], y[i], up ? 32 - s : s) & ~keep);
        }
    }
}
__device__ __forceinline__ uint32_t transpose32(uint32_t w, int lane) {
    uint32_t a[1] = {w};
    transpose32(a, lane);
    return a[0];
}

// Masks of rank bits 4k .. 4k + 3 of a unit node (tree_layout.h): the byte's top bit, after a
// shift by k, spread over the word.
__device__ __forceinline__ void rank_masks(uint32_t rank, int k, uint32_t (&m)[4]) {
    const uint32_t r = rank << k;
    asm("prmt.b32 %0, %1, 0, 0x8888;" : "=r"(m[0]) : "r"(r));
    asm("prmt.b32 %0, %1, 0, 0x9999;" : "=r"(m[1]) : "r"(r));
    asm("prmt.b32 %0, %1, 0, 0xAAAA;" : "=r"(m[2]) : "r"(r));
    asm("prmt.b32 %0, %1, 0, 0xBBBB;" : "=r"(m[3]) : "r"(r));
}

// Four more code bits of a sliced comparison (tree_layout.h): le for 32 rows.
__device__ __forceinline__ uint32_t slice_le(uint32_t le, const uint4 &q, const uint32_t (&m)[4]) {
    auto maj = [](uint32_t c, uint32_t mm, uint32_t l) { return (~c & mm) | (~c & l) | (mm & l); };
    return maj(q.w, m[3], maj(q.z, m[2], maj(q.y, m[1], maj(q.x, m[0], le))));
}

// Decisions of a unit node for the 32 rows of a code block (quads at `block`).
__device__ __forceinline__ uint32_t unit_decide(const uint2 &node, const uint4 *block, const SliceArrays &sa) {
    const int col = unit_column(node.x), nq = unit_quads(node.x);
    uint32_t le = 0u - unit_start(node.x), m[4];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (k < nq) {
            rank_masks(node.y, k, m);
            le = slice_le(le, block[sa.qbase[k] + col], m);
        }
    }
    return le;
}

// Rows with pattern p at leaf q = 4s + j of tree t: the leaf pattern p has the subtree-root
// pattern in its high D-2 bits, then the bit for node r and the bit for the child of r on the
// path; the decision at the other child of r is summed out.
__device__ __forceinline__ uint32_t leaf_count(int D, const uint32_t *__restrict__ hist, int leaf, uint32_t p) {
    const int t = leaf >> D, q = leaf & ((1 << D) - 1);
    const int s = q >> 2, j = q & 3;
    const int NS = 1 << (D - 2), E = 1 << (D + 1);
    const uint32_t pp = p >> 2, fn = (p >> 1) & 1u, fc = p & 1u;
    const uint32_t dn = (j < 2) ? fn : (fn ^ 1u);         // path goes left at r for j < 2
    const uint32_t dch = ((j & 1) == 0) ? fc : (fc ^ 1u);  // and left at the child for even j
    const uint32_t *h = hist + ((size_t)t * NS + s) * E;
    const uint32_t R = pp ^ (uint32_t)s;  // ancestors' raw decisions (wdf_internal.h)
    uint32_t e0, e1;
    if (j < 2) {  // the path takes 2r+1 (entry bit 0); sum over the decision at 2r+2
        e0 = (R << 3) | (dn << 2) | dch;
        e1 = e0 | 2u;
    } else {  // the path takes 2r+2 (entry bit 1); sum over the decision at 2r+1
        e0 = (R << 3) | (dn << 2) | (dch << 1);
        e1 = e0 | 1u;
    }
    return __ldg(h + e0) + __ldg(h + e1);
}

// Folded pair values (depth <= 6) of a bottom subtree with slots 0..D-3 = the ancestors of its
// root r (root first), D-2 = r, D-1 and D = r's children: every slot pair (u, v), u < v, except
// the two children (never on one path): iv_fp(D) values, padded to a multiple of 4.
__host__ __device__ constexpr int iv_fp(int D) { return (D + 1) * D / 2 - 1; }
__host__ __device__ constexpr int iv_fpp(int D) { return (iv_fp(D) + 3) & ~3; }
// index of slot pair (u, v), u < v, in a folded vector (pairs ordered by u, then v)
__host__ __device__ constexpr int iv_pidx(int D, int u, int v) {
    return u * D - u * (u - 1) / 2 + (v - u - 1);
}

// Decision code of value x in code column c (tree_layout.h).
__device__ __forceinline__ int decision_code(float x, const SliceArrays &sa, int c) {
    if (x != x) return __ldg(&sa.col[c].count);
    const int2 pk = __ldg(reinterpret_cast<const int2 *>(sa.pack) + (c >> 3));  // first, levels
    const float *tree = sa.thr + pk.x + ((c & 7) << pk.y);
    int i = 1;
    for (int l = 0; l < pk.y; ++l) i = 2 * i + (__ldg(tree + i) <= x ? 1 : 0);
    return i - (1 << pk.y);
}

}  // namespace wdf
