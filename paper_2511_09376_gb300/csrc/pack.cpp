// Host-side validation and complete-layout packing of a tree ensemble.
//
// Input format: Def. "decision_tree" (binary inner nodes with feature and threshold,
// leaves with outputs).  The complete layout and why it changes no value are
// described in wdf_internal.h.  Leaves are grouped by the path signature of section
// "Algorithmic Improvements" item 2 (the pattern-pair matrices depend only on the
// path length and on which features repeat along the path), so each group shares one
// pattern-pair table.
#include <algorithm>
#include <cstring>
#include <limits>
#include <map>

#include "tree_layout.h"
#include "wdf_internal.h"

namespace wdf {

namespace {

struct Src {
    int F;
    const int64_t *off;
    const int32_t *feat;
    const float *thr;
    const int32_t *left, *right;
    const float *val;
};

// Writes the subtree of input node `node` (local to tree t) at heap position h of
// depth `depth`; pass-through when node < 0 ("send left") and `keep` says whether the
// leftmost leaf below keeps output w.  csrc: the input node whose cover a pass-through
// position carries (the pushed-down leaf on the kept path, -1 elsewhere).
void place(const Src &s, int t, int32_t node, int h, int depth, float w, bool keep, Packed *p, int32_t csrc) {
    const int D = p->D;
    p->heap_src[(size_t)t * (p->NI + p->NL) + h] = (node >= 0) ? node : csrc;
    if (depth == D) {
        const int q = h - p->NI;
        p->leaf_w[(size_t)t * p->NL + q] = (node >= 0) ? s.val[s.off[t] + node] : (keep ? w : 0.0f);
        return;
    }
    const size_t k = (size_t)t * p->NI + h;
    if (node >= 0 && s.feat[s.off[t] + node] >= 0) {
        const int64_t g = s.off[t] + node;
        p->node_feat[k] = s.feat[g];
        p->node_thr[k] = s.thr[g];
        place(s, t, s.left[g], 2 * h + 1, depth + 1, 0.0f, false, p, -1);
        place(s, t, s.right[g], 2 * h + 2, depth + 1, 0.0f, false, p, -1);
        return;
    }
    // an input leaf above depth D, or a node under a pass-through: route every row left
    float wl = w;
    bool kl = keep;
    int32_t cl = csrc;
    if (node >= 0) {  // input leaf: its output (and cover) move to the leftmost leaf below
        wl = s.val[s.off[t] + node];
        kl = true;
        cl = node;
    }
    p->node_feat[k] = p->F;  // virtual column, always 0
    p->node_thr[k] = 1.0f;   // 0 < 1: left
    place(s, t, -1, 2 * h + 1, depth + 1, wl, kl, p, cl);
    place(s, t, -1, 2 * h + 2, depth + 1, 0.0f, false, p, -1);
}

// Decision codes, node records and tree metadata (tree_layout.h): columns sorted by width
// and grouped into packs, their search trees, the nodes of every unit, the real inner nodes
// and the flush order's features and batch flags.
void build_records(Packed *pp) {
    Packed &p = *pp;
    const int F = p.F, T = p.T, D = p.D, NI = p.NI;
    constexpr int cap = (1 << kSliceBits) - 1;  // thresholds of one column
    std::vector<std::vector<float>> thr((size_t)F);
    for (size_t k = 0; k < p.node_feat.size(); ++k) {
        const int f = p.node_feat[k];
        if (f < F && p.node_thr[k] == p.node_thr[k]) thr[(size_t)f].push_back(p.node_thr[k]);
    }
    struct Col {
        int f, lo, cnt, levels;
    };
    std::vector<Col> cols;
    for (int f = 0; f < F; ++f) {
        auto &v = thr[(size_t)f];
        std::sort(v.begin(), v.end());
        v.erase(std::unique(v.begin(), v.end(), [](float a, float b) { return a == b; }), v.end());
        for (int lo = 0; lo < (int)v.size(); lo += cap) {
            const int cnt = std::min((int)v.size() - lo, cap);
            cols.push_back(Col{f, lo, cnt, ilog2(cnt) + 1});
        }
    }
    if (cols.empty()) cols.push_back(Col{0, 0, 0, 1});  // no real threshold at all: one empty column
    std::stable_sort(cols.begin(), cols.end(), [](const Col &a, const Col &b) { return a.levels > b.levels; });
    while (cols.size() % 8) cols.push_back(Col{0, 0, 0, 1});
    // column of the j-th threshold of feature f: at[f][j / cap]
    std::vector<std::vector<int>> at((size_t)F);
    p.scol.clear();
    p.spack.clear();
    p.sgroup.clear();
    p.sthr.clear();
    int wide[3] = {0, 0, 0};
    for (size_t c0 = 0; c0 < cols.size(); c0 += 8) {
        const int levels = cols[c0].levels;  // the widest of the pack
        const int first = (int)p.sthr.size();
        for (int k = 0; k < 3; ++k)
            if (levels > 4 * k) wide[k] += 8;
        p.sthr.resize(p.sthr.size() + ((size_t)8 << levels), std::numeric_limits<float>::quiet_NaN());
        for (int j = 0; j < 8; ++j) {
            const Col &c = cols[c0 + (size_t)j];
            float *tree = p.sthr.data() + first + ((size_t)j << levels);
            const float *src = c.cnt ? thr[(size_t)c.f].data() + c.lo : nullptr;
            for (int i = 1; i < (1 << levels); ++i) {  // the threshold in the middle of node i's range
                int d = ilog2(i);
                const int rank = ((i - (1 << d)) << (levels - d)) + (1 << (levels - d - 1)) - 1;
                if (rank < c.cnt) tree[i] = src[rank];
            }
            if (c.cnt) {
                auto &a = at[(size_t)c.f];
                if ((int)a.size() <= c.lo / cap) a.resize((size_t)(c.lo / cap + 1), 0);
                a[(size_t)(c.lo / cap)] = (int)(c0 + (size_t)j);
            }
            p.scol.push_back(SliceCol{c.f, c.cnt});
        }
        p.spack.push_back(SlicePack{first, levels});
        const int pack = (int)p.spack.size() - 1, size = 8 << levels;
        if (p.sgroup.empty() || p.sgroup.back().thr_n + size > kSliceGroupFloats ||
            pack - p.sgroup.back().pack0 >= kSliceGroupPacks)
            p.sgroup.push_back(SliceGroup{pack, pack, first, 0});
        p.sgroup.back().pack1 = pack + 1;
        p.sgroup.back().thr_n += size;
    }
    p.qbase[0] = 0;
    p.qbase[1] = wide[0];
    p.qbase[2] = wide[0] + wide[1];
    p.quads = wide[0] + wide[1] + wide[2];
    // per complete-layout node: its column and rank (-1: pass-through, or a NaN threshold)
    std::vector<int32_t> col((size_t)T * NI, -1), rank((size_t)T * NI, -1);
    for (size_t k = 0; k < col.size(); ++k) {
        const int f = p.node_feat[k];
        const float x = p.node_thr[k];
        if (f == F || x != x) continue;
        const auto &s = thr[(size_t)f];
        const int j = (int)(std::lower_bound(s.begin(), s.end(), x) - s.begin());
        col[k] = at[(size_t)f][(size_t)(j / cap)];
        rank[k] = j % cap;
    }
    const int U = units_per_tree(D), n_local = (1 << unit_height(D)) - 1, FL = flush_len(D);
    std::vector<int> lane_node((size_t)U * 32, -1), pos_node((size_t)FL);
    for (int u = 0; u < U; ++u)
        for (int i = 0; i < 32; ++i)
            lane_node[(size_t)u * 32 + i] = i < n_local ? unit_node(D, u, i) : (i == 31 && u < U - 1 ? u : -1);
    for (int i = 0; i < FL; ++i) pos_node[(size_t)i] = flush_node(D, i);
    p.unit.assign((size_t)T * U * 32, UnitNode{0u, 0u});
    p.rec.assign((size_t)T * NI, NodeRec{0, -1, 0u, 0u});
    p.meta.assign((size_t)T, TreeMeta{});
    p.flush_feat.assign((size_t)T * FL, F);
    p.flush_rep.assign((size_t)T * (FL / 8), 0);
    for (int t = 0; t < T; ++t) {
        const int32_t *feat = &p.node_feat[(size_t)t * NI], *tc = &col[(size_t)t * NI], *tr = &rank[(size_t)t * NI];
        for (int i = 0; i < U * 32; ++i) {
            const int v = lane_node[(size_t)i];
            if (v < 0) continue;
            UnitNode &n = p.unit[(size_t)t * U * 32 + i];
            if (feat[v] == F) {
                n.at = unit_at(0u, 0u, 1u);  // pass-through: always left
            } else if (tc[v] >= 0) {
                const int levels = p.spack[(size_t)(tc[v] / 8)].levels;
                n.at = unit_at((uint32_t)tc[v], (uint32_t)((levels + 3) / 4), 1u);  // at most kMostColumns: api.cu
                for (int b = 0; b < kSliceBits; ++b)
                    if ((tr[v] >> b) & 1) n.rank |= (0x80u >> (b / 4)) << (8 * (b % 4));
            }  // a NaN threshold: never left
        }
        TreeMeta &m = p.meta[(size_t)t];
        int c = 0;
        for (int v = 0; v < NI; ++v) {  // heap order, so the nodes of word v/32 are contiguous
            if (feat[v] == F)
                m.pt[v >> 5] |= 1u << (v & 31);
            else
                p.rec[(size_t)t * NI + c++] =
                    NodeRec{tc[v] >= 0 ? tc[v] : 0, tr[v], (D >= 7 || v < 32) ? 1u << (v & 31) : 0u,
                            (D <= 6 && v >= 32) ? 1u << (v - 32) : 0u};
            if ((v & 31) == 31 || v == NI - 1) m.wend[v >> 5] = (uint8_t)c;
        }
        for (int w = (NI - 1) / 32 + 1; w < 8; ++w) m.wend[w] = (uint8_t)c;
        m.live = p.live[(size_t)t];
        for (int b = 0; b < flush_batches(D); ++b) {
            uint32_t rep = 0;
            bool real = false, again = false;
            for (int i = 8 * b; i < 8 * b + 8; ++i) {
                const int v = pos_node[(size_t)i];
                if (v < 0 || feat[v] == F) continue;  // pass-through nodes all write the scratch row
                p.flush_feat[(size_t)t * FL + i] = feat[v];
                real = true;
                for (int j = 8 * b; j < i; ++j)
                    if (pos_node[(size_t)j] >= 0 && feat[pos_node[(size_t)j]] == feat[v]) {
                        again = again || ((rep >> (j - 8 * b)) & 1u);
                        rep |= 1u << (i - 8 * b);
                    }
            }
            if (!rep) m.flush |= 1ull << b;
            p.flush_rep[(size_t)t * (FL / 8) + b] = (uint8_t)(again ? 0xFFu : rep);
            if (real) m.real |= 1ull << b;
        }
    }
}

// The nodes of every feature in the order of the consumer kernel (k_explain.cuh): within a part
// its trees two by two, in turns unit by unit; within a unit its flush positions; the nodes
// above the units with the tree's last unit.
void build_value_lists(Packed *pp) {
    Packed &p = *pp;
    const int F = p.F, T = p.T, D = p.D, FL = flush_len(D), GL = flush_group_len(D), U = units_per_tree(D);
    const int P = explain_parts(T, D);
    p.voff.assign((size_t)F * P + 1, 0);
    std::vector<int32_t> count((size_t)F * P + 1, 0);
    for (int pass = 0; pass < 2; ++pass) {
        for (int part = 0; part < P; ++part) {
            const int tb = (int)((long long)T * part / P), te = (int)((long long)T * (part + 1) / P);
            for (int t0 = tb; t0 < te; t0 += 2)
                for (int u = 0; u < U; ++u)
                    for (int t = t0; t < te && t < t0 + 2; ++t) {
                        const int end = u == U - 1 ? FL : (u + 1) * GL;
                        for (int i = u * GL; i < end; ++i) {
                            const int f = p.flush_feat[(size_t)t * FL + i];
                            if (f == F) continue;
                            const size_t k = (size_t)f * P + part;
                            if (pass == 0) ++p.voff[k + 1];
                            else p.vlist[(size_t)p.voff[k] + count[k]++] = t * FL + i;
                        }
                    }
        }
        if (pass == 0) {
            for (size_t k = 0; k < (size_t)F * P; ++k) p.voff[k + 1] += p.voff[k];
            p.vlist.assign((size_t)p.voff[(size_t)F * P], 0);
        }
    }
}

}  // namespace

int pack_ensemble(int F, int T, const int64_t *off, const int32_t *feat, const float *thr, const int32_t *left,
                  const int32_t *right, const float *val, Packed *out, std::string *err) {
    if (F < 1 || T < 1 || !off || !feat || !thr || !left || !right || !val) {
        *err = "n_features and n_trees must be >= 1 and all arrays non-null";
        return 1;
    }
    if (off[0] != 0) {
        *err = "tree_offset[0] must be 0";
        return 1;
    }
    int max_depth = 0;
    std::vector<int> depth_of, seen;
    for (int t = 0; t < T; ++t) {
        const int64_t o = off[t], sz = off[t + 1] - off[t];
        if (sz < 1 || sz > (1 << 20)) {
            *err = "tree " + std::to_string(t) + ": node count must be in [1, 2^20]";
            return 1;
        }
        depth_of.assign((size_t)sz, -1);
        seen.assign((size_t)sz, 0);
        std::vector<int32_t> queue;
        queue.push_back(0);
        depth_of[0] = 0;
        seen[0] = 1;
        size_t head = 0;
        while (head < queue.size()) {
            const int32_t v = queue[head++];
            const int64_t g = o + v;
            if (feat[g] < 0) {
                max_depth = std::max(max_depth, depth_of[(size_t)v]);
                continue;
            }
            if (feat[g] >= F) {
                *err = "tree " + std::to_string(t) + " node " + std::to_string(v) + ": feature out of range";
                return 1;
            }
            for (int32_t c : {left[g], right[g]}) {
                if (c <= 0 || c >= sz) {
                    *err = "tree " + std::to_string(t) + " node " + std::to_string(v) + ": child index out of range";
                    return 1;
                }
                if (seen[(size_t)c]) {
                    *err = "tree " + std::to_string(t) + " node " + std::to_string(c) + ": reached twice";
                    return 1;
                }
                seen[(size_t)c] = 1;
                depth_of[(size_t)c] = depth_of[(size_t)v] + 1;
                if (depth_of[(size_t)c] > kMaxDepth) {
                    *err = "tree " + std::to_string(t) + ": depth above 8 is not supported";
                    return 4;
                }
                queue.push_back(c);
            }
        }
        if ((int64_t)queue.size() != sz) {
            *err = "tree " + std::to_string(t) + ": " + std::to_string(sz - (int64_t)queue.size()) +
                   " node(s) not reachable from the root";
            return 1;
        }
    }
    Packed &p = *out;
    p = Packed();
    p.F = F;
    p.T = T;
    p.D = std::max(kMinDepth, max_depth);
    p.NI = (1 << p.D) - 1;
    p.NL = 1 << p.D;
    p.NS = 1 << (p.D - 2);
    p.node_feat.assign((size_t)T * p.NI, 0);
    p.node_thr.assign((size_t)T * p.NI, 0.0f);
    p.leaf_w.assign((size_t)T * p.NL, 0.0f);
    p.live.assign((size_t)T, 0);
    p.leaf_row.assign((size_t)T * p.NL, -1);
    p.heap_src.assign((size_t)T * (p.NI + p.NL), -1);
    p.in_off.assign(off, off + T + 1);
    Src s{F, off, feat, thr, left, right, val};
    for (int t = 0; t < T; ++t) place(s, t, 0, 0, 0, 0.0f, false, &p, -1);

    // live bottom subtrees and signature groups of the live leaves
    std::map<uint32_t, std::vector<int32_t>> groups;
    const int D = p.D;
    for (int t = 0; t < T; ++t) {
        for (int q = 0; q < p.NL; ++q) {
            if (p.leaf_w[(size_t)t * p.NL + q] == 0.0f) continue;
            p.live[(size_t)t] |= (uint64_t)1 << (q >> 2);
            int32_t pf[kMaxDepth];
            uint32_t key = 0;
            for (int k = 0; k < D; ++k) {
                const int h = ((p.NL + q) >> (D - k)) - 1;  // heap index of the depth-k node on the path
                const int32_t f = p.node_feat[(size_t)t * p.NI + h];
                pf[k] = (f == F) ? -(k + 1) : f;  // pass-through positions never repeat
                int first = k;
                for (int j = 0; j < k; ++j)
                    if (pf[j] == pf[k]) { first = j; break; }
                key |= (uint32_t)first << (3 * k);
            }
            groups[key].push_back(t * p.NL + q);
        }
    }
    p.group_off.push_back(0);
    for (auto &kv : groups) {
        p.sig_key.push_back(kv.first);
        for (int32_t leaf : kv.second) {
            p.leaf_row[(size_t)leaf] = (int32_t)p.group_leaf.size();
            p.group_leaf.push_back(leaf);
        }
        p.group_off.push_back((int32_t)p.group_leaf.size());
    }
    build_records(&p);
    build_value_lists(&p);
    return 0;
}

int pd_ratios(const Packed &p, const double *cover, std::vector<double> *ratio, std::string *err) {
    if (!cover) {
        *err = "cover is null";
        return 1;
    }
    const int64_t total = p.in_off[(size_t)p.T];
    for (int64_t i = 0; i < total; ++i)
        if (!(cover[i] >= 0.0) || cover[i] > 1e300) {
            *err = "covers must be finite and non-negative (node " + std::to_string(i) + ")";
            return 1;
        }
    const int D = p.D;
    ratio->assign(p.group_leaf.size() * (size_t)D, 0.0);
    for (size_t row = 0; row < p.group_leaf.size(); ++row) {
        const int leaf = p.group_leaf[row];
        const int t = leaf / p.NL, q = leaf % p.NL;
        auto cov = [&](int h) {
            const int32_t src = p.heap_src[(size_t)t * (p.NI + p.NL) + h];
            return src >= 0 ? cover[p.in_off[(size_t)t] + src] : 0.0;
        };
        for (int k = 0; k < D; ++k) {
            const int h = ((p.NL + q) >> (D - k)) - 1;          // path node at depth k
            const int hn = ((p.NL + q) >> (D - k - 1)) - 1;     // the next one on the path
            if (p.node_feat[(size_t)t * p.NI + h] == p.F) {      // pass-through: every row goes left
                (*ratio)[row * D + k] = 1.0;
                continue;
            }
            const double cn = cov(h);
            (*ratio)[row * D + k] = cn > 0.0 ? cov(hn) / cn : 0.0;
        }
    }
    return 0;
}

}  // namespace wdf
