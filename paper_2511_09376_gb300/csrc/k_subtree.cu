// Steps 2 and 3 of Algorithm 3 for background counts in FP32, per bottom subtree: the slot
// vectors the consumer kernel gathers, straight from the joint entry counts.
//
// For one leaf let the variables be the distinct features on its path.  A row with pattern p
// "keeps" variable i when it follows the path at every position of i.  The cube of a consumer
// that keeps the set S and a background row that keeps all but the set Z is satisfiable
// exactly when Z is part of S (rules 1-4 of section "Constructing a WDNF Representation": a
// position both leave makes the cube empty, and a variable that appears both plain and
// negated drops it); then its positive literals are Z, its negative ones the complement of S.
// With a = |Z| and b = the number of variables outside S its values (Formulas
// "shap_simplified_formula", "banzhaf_simplified_formula") depend on a and b alone, so with
//   G[a][S] = the number of background rows with Z in S and |Z| = a,
// a subset sum over the exact integer counts (D additions per element),
//   value of i outside S:  sum_a vneg(a, b) G[a][S]
//   value of i in S:       sum_a vpos(a, b) (G[a][S] - G[a][S without i])   (i in Z),
// the difference exact in integers and all terms of one sign.  A leaf of depth 8 takes some
// 20,000 additions and multiplications where its dense 256 x 2048 table takes 524,288
// multiply-adds; the FP32 error is that of a handful of terms instead of 256.
//
// A block takes one bottom subtree: its four leaves' counts, subset sums and values in shared
// memory, then the entries (k_fold of k_contract.cu: slots above the subtree and its root from
// all four leaves, its children from two each), so no per-leaf value goes to memory.  Bound by
// shared-memory wavefronts, half of them the subset sums, half the loads of the values (about
// 7,000 per subtree of depth 8, 9,400 clocks).  300 trees of depth 8: 578 us, where per-leaf
// counts, the dense contraction and the fold took 45 + 2125 + 263.
#include "launch.h"
#include "wdf_device.cuh"

namespace wdf {

namespace {
struct CubeValues {
    float pos[9][9], neg[9][9];  // [a][b]
};

CubeValues cube_values(int metric) {
    CubeValues v;
    double fact[9] = {1, 1, 2, 6, 24, 120, 720, 5040, 40320};
    for (int a = 0; a < 9; ++a)
        for (int b = 0; b < 9; ++b) {
            double p = 0.0, n = 0.0;
            if (a + b <= 8) {
                if (metric == 1) {
                    p = a > 0 ? 1.0 / (double)(1 << (a + b - 1)) : 0.0;
                    n = b > 0 ? -1.0 / (double)(1 << (a + b - 1)) : 0.0;
                } else {
                    p = a > 0 ? fact[a - 1] * fact[b] / fact[a + b] : 0.0;
                    n = b > 0 ? -fact[a] * fact[b - 1] / fact[a + b] : 0.0;
                }
            }
            v.pos[a][b] = (float)p;
            v.neg[a][b] = (float)n;
        }
    return v;
}
}  // namespace

template <int D>
struct SubtreeCfg {
    static constexpr int K = 1 << D, THREADS = D >= 7 ? 256 : 128;
    static constexpr size_t SUMS = (size_t)4 * (D + 1) * K * 4;  // four leaves' subset sums
};

// What the four leaves of a bottom subtree share out: per leaf the bit of every position's
// variable (the bit of the feature's first position), the variables' bits, and w / m.
template <int D>
struct SubtreeLeaves {
    uint32_t keep[4][D], act[4];
    float fac[4];

    // the variables that pattern p of leaf j keeps
    __device__ __forceinline__ uint32_t kept(int j, uint32_t p) const {
        uint32_t set = act[j];
#pragma unroll
        for (int k = 0; k < D; ++k)
            if (!((p >> (D - 1 - k)) & 1u)) set &= ~keep[j][k];
        return set;
    }
};

// G[leaf][a][S] of the block's subtree (all threads of the block; ends synchronised).
template <int D>
__device__ __forceinline__ void subtree_sums(SubtreeLeaves<D> &lv, uint32_t *G, const uint32_t *__restrict__ h,
                                             const int2 *__restrict__ tree_nodes, int F,
                                             const int32_t *__restrict__ tree_leaf_row,
                                             const float *__restrict__ scale, int s) {
    using S = Shape<D>;
    constexpr int K = SubtreeCfg<D>::K, NT = SubtreeCfg<D>::THREADS;
    const int tid = threadIdx.x;
    if (tid < 4) {
        const int q = 4 * s + tid, row = __ldg(tree_leaf_row + q);
        int feat[D];
        uint32_t a = 0u;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            feat[k] = __ldg(&tree_nodes[((S::NL + q) >> (D - k)) - 1].x);
            int first = k;
#pragma unroll
            for (int j = k - 1; j >= 0; --j)
                if (feat[j] == feat[k] && feat[k] != F) first = j;  // pass-through positions never repeat
            lv.keep[tid][k] = 1u << (D - 1 - first);
            a |= lv.keep[tid][k];
        }
        lv.act[tid] = a;
        lv.fac[tid] = row >= 0 ? __ldg(scale + row) : 0.0f;
    }
    for (int i = tid; i < 4 * (D + 1) * K; i += NT) G[i] = 0u;
    __syncthreads();
    for (int i = tid; i < 4 * K; i += NT) {
        const int j = i >> D;
        const uint32_t p = (uint32_t)i & (K - 1);
        const uint32_t fn = (p >> 1) & 1u, fc = p & 1u, dn = j < 2 ? fn : fn ^ 1u, dc = (j & 1) ? fc ^ 1u : fc;
        const uint32_t e0 = ((((p >> 2) ^ (uint32_t)s) << 3) | (dn << 2)) | (j < 2 ? dc : dc << 1);
        const uint32_t c = __ldg(h + e0) + __ldg(h + (e0 | (j < 2 ? 2u : 1u)));
        const uint32_t z = lv.act[j] & ~lv.kept(j, p);
        if (c) atomicAdd(&G[(j * (D + 1) + __popc(z)) * K + z], c);
    }
#pragma unroll 1
    for (int b = 0; b < D; ++b) {  // subset sums over every bit
        __syncthreads();
        for (int i = tid; i < 4 * (D + 1) * (K / 2); i += NT) {
            const uint32_t x = (uint32_t)i & (K / 2 - 1), y = (uint32_t)i >> (D - 1);
            const uint32_t m = ((x >> b) << (b + 1)) | (x & ((1u << b) - 1u));
            G[y * K + (m | (1u << b))] += G[y * K + m];
        }
    }
    __syncthreads();
}

template <int D>
__global__ void __launch_bounds__(SubtreeCfg<D>::THREADS) k_subtree_fold(const uint32_t *__restrict__ hist,
                                                                        const int2 *__restrict__ nodes, int F,
                                                                        const int32_t *__restrict__ leaf_row,
                                                                        const float *__restrict__ scale, int T,
                                                                        const uint32_t *__restrict__ lines,
                                                                        float *__restrict__ sfold, CubeValues cv) {
    using S = Shape<D>;
    constexpr int K = SubtreeCfg<D>::K, NT = SubtreeCfg<D>::THREADS, X1 = extra_slots(D), SP = S::SP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *G = reinterpret_cast<uint32_t *>(smem_raw);                       // [leaf][a][set]
    float *V = reinterpret_cast<float *>(smem_raw + SubtreeCfg<D>::SUMS);       // [leaf][position][pattern]
    __shared__ SubtreeLeaves<D> lv;
    __shared__ float vpos[(D + 1) * (D + 1)], vneg[(D + 1) * (D + 1)];
    const int tid = threadIdx.x, t = blockIdx.x / S::NS, s = blockIdx.x % S::NS;
    const int64_t sub = (int64_t)t * S::NS + s;
    const uint32_t rot = (__ldg(lines + (size_t)t * lines_words(D) + (s >> 2)) >> (8 * (s & 3))) & 0xFFu;
    float *extra = sfold + (int64_t)T * S::NS * S::E * SP + sub * S::E;
    if (rot == kLineDead) {  // dead: every row reads entry 0
        if (tid < SP) sfold[sub * S::E * SP + tid] = 0.0f;
        if (X1 && tid == 0) extra[0] = 0.0f;
        return;
    }
    for (int i = tid; i < (D + 1) * (D + 1); i += NT) {
        vpos[i] = cv.pos[i / (D + 1)][i % (D + 1)];
        vneg[i] = cv.neg[i / (D + 1)][i % (D + 1)];
    }
    subtree_sums<D>(lv, G, hist + sub * S::E, nodes + (size_t)t * S::NI, F, leaf_row + (size_t)t * S::NL, scale, s);
    for (int i = tid; i < 4 * K; i += NT) {
        const int j = i >> D;
        const uint32_t p = (uint32_t)i & (K - 1), set = lv.kept(j, p);
        const int b = __popc(lv.act[j]) - __popc(set);
        const uint32_t *g = G + (size_t)j * (D + 1) * K;
        uint32_t all[D + 1];
        float minus = 0.0f;
#pragma unroll
        for (int a = 0; a <= D; ++a) {
            all[a] = g[a * K + set];
            if (a + b <= D) minus = fmaf(vneg[a * (D + 1) + b], (float)all[a], minus);
        }
        float *out = V + (size_t)j * D * K + p;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const uint32_t bit = 1u << (D - 1 - k);
            float x = 0.0f;
            if (lv.act[j] & bit) {
                if (set & bit) {
#pragma unroll
                    for (int a = 1; a <= D; ++a)
                        if (a + b <= D)
                            x = fmaf(vpos[a * (D + 1) + b], (float)(all[a] - g[a * K + (set ^ bit)]), x);
                } else {
                    x = minus;
                }
            }
            out[k * K] = x * lv.fac[j];
        }
    }
    __syncthreads();
    for (int e = tid; e < S::E; e += NT) {
        const uint32_t pp = ((uint32_t)e >> 3) ^ (uint32_t)s, dn = (e >> 2) & 1, dnl = e & 1, dnr = (e >> 1) & 1;
        float o[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) o[k] = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t fn = j < 2 ? dn : dn ^ 1u, dch = j < 2 ? dnl : dnr, fc = (j & 1) == 0 ? dch : dch ^ 1u;
            const float *vj = V + (size_t)j * D * K + ((pp << 2) | (fn << 1) | fc);
#pragma unroll
            for (int k = 0; k <= D - 2; ++k) o[k] += vj[k * K];
            o[j < 2 ? D - 1 : D] += vj[(D - 1) * K];
        }
        const uint32_t at = line_pos((uint32_t)e, rot, D);
        float4 *dst = reinterpret_cast<float4 *>(sfold + (sub * S::E + at) * SP);
#pragma unroll
        for (int k = 0; k < SP; k += 4) dst[k / 4] = make_float4(o[k + X1], o[k + 1 + X1], o[k + 2 + X1], o[k + 3 + X1]);
        if (X1) extra[at] = o[0];
    }
}

// The pairs: a row keeps or drops each of two variables, so the cube's pair value (Table
// "table_shap_iv", Formula "banzhaf_simplified_formula_interactions") has three cases, again
// by a and b alone:
//   both outside S:  sum_a nn(a, b) G[a][S]
//   i in S, j not:   sum_a pn(a, b) (G[a][S] - G[a][S - i])
//   both in S:       sum_a pp(a, b) (G[a][S] - G[a][S - i] - G[a][S - j] + G[a][S - i - j]).
// One load per pair and a; the differences to S - i are kept for all i.  Depth <= 6 folds the
// four leaves per entry, deeper trees store each live leaf's vector.  200 trees of depth 6: 45 us,
// where pair tables, their contraction and the fold took 32 + 61 + 56.
struct PairValues {
    float pp[9][9], pn[9][9], nn[9][9];  // [a][b]
};

static PairValues pair_values(int metric) {
    PairValues v;
    const double fact[9] = {1, 1, 2, 6, 24, 120, 720, 5040, 40320};
    for (int a = 0; a < 9; ++a)
        for (int b = 0; b < 9; ++b) {
            double pp = 0.0, pn = 0.0, nn = 0.0;
            const int s = a + b;
            if (s >= 2 && s <= 8) {
                if (metric == 1) {
                    const double x = 1.0 / (double)(1 << (s - 2));
                    if (a >= 2) pp = x;
                    if (b >= 2) nn = x;
                    if (a >= 1 && b >= 1) pn = -x;
                } else {
                    if (a >= 2) pp = fact[a - 2] * fact[b] / fact[s - 1];
                    if (b >= 2) nn = fact[b - 2] * fact[a] / fact[s - 1];
                    if (a >= 1 && b >= 1) pn = -fact[a - 1] * fact[b - 1] / fact[s - 1];
                }
            }
            v.pp[a][b] = (float)pp;
            v.pn[a][b] = (float)pn;
            v.nn[a][b] = (float)nn;
        }
    return v;
}

template <int D>
__global__ void __launch_bounds__(SubtreeCfg<D>::THREADS) k_subtree_pairs(const uint32_t *__restrict__ hist,
                                                                         const int2 *__restrict__ nodes, int F,
                                                                         const int32_t *__restrict__ leaf_row,
                                                                         const float *__restrict__ scale,
                                                                         const TreeMeta *__restrict__ meta,
                                                                         float *__restrict__ out, PairValues pv) {
    using S = Shape<D>;
    constexpr int K = SubtreeCfg<D>::K, NT = SubtreeCfg<D>::THREADS, P = D * (D - 1) / 2, PP = (P + 3) & ~3;
    constexpr bool FOLD = D <= 6;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *G = reinterpret_cast<uint32_t *>(smem_raw);                  // [leaf][a][set]
    float *V = reinterpret_cast<float *>(smem_raw + SubtreeCfg<D>::SUMS);  // FOLD: [leaf][pair][pattern]
    __shared__ SubtreeLeaves<D> lv;
    __shared__ float vpp[(D + 1) * (D + 1)], vpn[(D + 1) * (D + 1)], vnn[(D + 1) * (D + 1)];
    const int tid = threadIdx.x, t = blockIdx.x / S::NS, s = blockIdx.x % S::NS;
    const int64_t sub = (int64_t)t * S::NS + s;
    if (!((__ldg(&meta[t].live) >> s) & 1ull)) return;  // no row reads a dead subtree
    for (int i = tid; i < (D + 1) * (D + 1); i += NT) {
        vpp[i] = pv.pp[i / (D + 1)][i % (D + 1)];
        vpn[i] = pv.pn[i / (D + 1)][i % (D + 1)];
        vnn[i] = pv.nn[i / (D + 1)][i % (D + 1)];
    }
    subtree_sums<D>(lv, G, hist + sub * S::E, nodes + (size_t)t * S::NI, F, leaf_row + (size_t)t * S::NL, scale, s);
    for (int i = tid; i < 4 * K; i += NT) {
        const int j = i >> D;
        const int row = __ldg(leaf_row + (size_t)t * S::NL + 4 * s + j);
        if (!FOLD && row < 0) continue;
        const uint32_t p = (uint32_t)i & (K - 1), set = lv.kept(j, p), act = lv.act[j];
        const int nset = __popc(set), b = __popc(act) - nset;
        const uint32_t *g = G + (size_t)j * (D + 1) * K;
        float both[P], one[D], none = 0.0f;
#pragma unroll
        for (int q = 0; q < P; ++q) both[q] = 0.0f;
#pragma unroll
        for (int k = 0; k < D; ++k) one[k] = 0.0f;
#pragma unroll 1
        for (int a = 0; a <= nset; ++a) {  // a + b <= number of variables
            const uint32_t *ga = g + a * K;
            const uint32_t all = ga[set];
            const float pp = vpp[a * (D + 1) + b], pn = vpn[a * (D + 1) + b];
            none = fmaf(vnn[a * (D + 1) + b], (float)all, none);
            uint32_t d[D];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const uint32_t bit = 1u << (D - 1 - k);
                d[k] = all - ga[set & ~bit];
                one[k] = fmaf(pn, (float)d[k], one[k]);
            }
            if (a >= 2) {
                int q = 0;
#pragma unroll
                for (int k1 = 0; k1 < D; ++k1)
#pragma unroll
                    for (int k2 = k1 + 1; k2 < D; ++k2, ++q) {
                        const uint32_t bits = (1u << (D - 1 - k1)) | (1u << (D - 1 - k2));
                        if ((set & bits) == bits)
                            both[q] = fmaf(pp, (float)(d[k1] + d[k2] - all + ga[set ^ bits]), both[q]);
                    }
            }
        }
        const float fac = lv.fac[j];
        float v[PP];
        int q = 0;
#pragma unroll
        for (int k1 = 0; k1 < D; ++k1)
#pragma unroll
            for (int k2 = k1 + 1; k2 < D; ++k2, ++q) {
                const uint32_t b1 = 1u << (D - 1 - k1), b2 = 1u << (D - 1 - k2);
                float x = 0.0f;
                if ((act & b1) && (act & b2))
                    x = (set & b1) ? ((set & b2) ? both[q] : one[k1]) : ((set & b2) ? one[k2] : none);
                v[q] = x * fac;
            }
#pragma unroll
        for (int k = P; k < PP; ++k) v[k] = 0.0f;
        if (FOLD) {
#pragma unroll
            for (int k = 0; k < P; ++k) V[((size_t)j * P + k) * K + p] = v[k];
        } else {
            float4 *dst = reinterpret_cast<float4 *>(out + ((size_t)row * K + p) * PP);
#pragma unroll
            for (int k = 0; k < PP; k += 4) dst[k / 4] = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
        }
    }
    if constexpr (FOLD) {
        constexpr int FPP = iv_fpp(D);
        __syncthreads();
        for (int e = tid; e < S::E; e += NT) {
            const uint32_t pp = ((uint32_t)e >> 3) ^ (uint32_t)s, dn = (e >> 2) & 1, dnl = e & 1, dnr = (e >> 1) & 1;
            float o[FPP];
#pragma unroll
            for (int k = 0; k < FPP; ++k) o[k] = 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t fn = j < 2 ? dn : dn ^ 1u, dch = j < 2 ? dnl : dnr, fc = (j & 1) == 0 ? dch : dch ^ 1u;
                const float *vj = V + (size_t)j * P * K + ((pp << 2) | (fn << 1) | fc);
                int q = 0;
#pragma unroll
                for (int k1 = 0; k1 < D; ++k1)
#pragma unroll
                    for (int k2 = k1 + 1; k2 < D; ++k2, ++q)
                        o[iv_pidx(D, k1, k2 == D - 1 && j >= 2 ? D : k2)] += vj[q * K];
            }
            float4 *dst = reinterpret_cast<float4 *>(out + (sub * S::E + e) * FPP);
#pragma unroll
            for (int k = 0; k < FPP; k += 4) dst[k / 4] = make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
        }
    }
}

template <int D>
static cudaError_t subtree_t(int metric, const uint32_t *hist, const int2 *nodes, int F, const int32_t *leaf_row,
                             const float *scale, int T, const uint32_t *lines, float *sfold, const DevInfo &dev,
                             cudaStream_t st) {
    constexpr size_t smem = SubtreeCfg<D>::SUMS + (size_t)4 * D * (1 << D) * 4;
    if (smem > dev.smem_optin) return cudaErrorInvalidConfiguration;
    auto kern = k_subtree_fold<D>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<(unsigned)(T * Shape<D>::NS), SubtreeCfg<D>::THREADS, smem, st>>>(hist, nodes, F, leaf_row, scale, T, lines,
                                                                           sfold, cube_values(metric));
    count_launches(1);
    return cudaGetLastError();
}

template <int D>
static cudaError_t pairs_t(int metric, const uint32_t *hist, const int2 *nodes, int F, const int32_t *leaf_row,
                           const float *scale, int T, const TreeMeta *meta, float *out, const DevInfo &dev,
                           cudaStream_t st) {
    constexpr size_t smem = SubtreeCfg<D>::SUMS + (D <= 6 ? (size_t)4 * (D * (D - 1) / 2) * (1 << D) * 4 : 0);
    if (smem > dev.smem_optin) return cudaErrorInvalidConfiguration;
    auto kern = k_subtree_pairs<D>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<(unsigned)(T * Shape<D>::NS), SubtreeCfg<D>::THREADS, smem, st>>>(hist, nodes, F, leaf_row, scale, meta, out,
                                                                           pair_values(metric));
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_subtree_fold(int D, int metric, const uint32_t *hist, const int2 *nodes, int F,
                                const int32_t *leaf_row, const float *scale, int T, const uint32_t *lines,
                                float *sfold, const DevInfo &dev, cudaStream_t st) {
    switch (D) {
        case 2: return subtree_t<2>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        case 3: return subtree_t<3>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        case 4: return subtree_t<4>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        case 5: return subtree_t<5>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        case 6: return subtree_t<6>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        case 7: return subtree_t<7>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        case 8: return subtree_t<8>(metric, hist, nodes, F, leaf_row, scale, T, lines, sfold, dev, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_subtree_pairs(int D, int metric, const uint32_t *hist, const int2 *nodes, int F,
                                 const int32_t *leaf_row, const float *scale, int T, const TreeMeta *meta,
                                 float *out, const DevInfo &dev, cudaStream_t st) {
    switch (D) {
        case 2: return pairs_t<2>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        case 3: return pairs_t<3>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        case 4: return pairs_t<4>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        case 5: return pairs_t<5>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        case 6: return pairs_t<6>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        case 7: return pairs_t<7>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        case 8: return pairs_t<8>(metric, hist, nodes, F, leaf_row, scale, T, meta, out, dev, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace wdf
