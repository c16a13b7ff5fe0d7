// Ragged batches: one graph launch explains requests against many ensembles of
// different depths and feature counts.
//
// Ensembles are grouped into classes by depth (one kernel instantiation each) and shared memory.  A
// call writes every class's work description -- the ensembles' device arrays (jobs),
// the requests, the encode items (request, group of columns, 32-row blocks) and the work items (job,
// request, first row, group of parts) of tile_rows consumer rows each -- into one pinned host blob; the
// captured graph copies that blob to the device with a single memcpy and then runs, per
// class on parallel branches, k_encode_batch (the rows' decision codes into the batch's
// code arena) and one persistent k_explain_batch.  The item count is read on the device, so the same graph serves
// every call until a capacity grows.  Results per consumer row are exactly those of
// wdf_explain: the per-row arithmetic and its order do not depend on the batch.
//
// The autotuner times every tile size that fits the class's shared-memory budget on the
// caller's own requests and keeps the fastest per class; results can be cached in a text
// file keyed by (depth, feature count rounded up to 32).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <sstream>
#include <string>
#include <vector>

#include "wdf_objects.h"
#include "woodelf.h"

namespace {

size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }

wdf_status fail(wdf_status s, const std::string &msg) {
    wdf::set_last_error(msg);
    return s;
}

#define WDF_CUDA(call)                                                                        \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess) return fail(WDF_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

struct Cls {
    int D = 0, room = 0, F_max = 0, q_max = 0, thr_max = 0, tile_rows = 0;
    bool wide = false;
    std::vector<int> members;  // batch ensemble indices, in job-slot order
    int cap_reqs = 0, cap_items = 0, cap_eitems = 0, cap_tiles = 0;
    size_t off_jobs = 0, off_reqs = 0, off_items = 0, off_count = 0, off_eitems = 0, off_ecount = 0;
};

// Rows of a request's code region: a multiple of every tile size (and of 32).
constexpr int64_t kCodePad = 128;
int64_t padded_rows(int64_t n) { return (n + kCodePad - 1) / kCodePad * kCodePad; }

// Most scratch of the parts of one call's split requests; kept until the batch is destroyed.
constexpr size_t kPartsBytes = (size_t)128 << 20;
constexpr int kMostItemBlocks = 16;  // 32-row blocks of an encode item

}  // namespace

struct wdf_batch {
    wdf_ctx *ctx = nullptr;
    std::vector<wdf_ensemble *> ens;
    std::vector<int> cls_of, slot_of;
    std::vector<Cls> cls;
    unsigned char *h_blob = nullptr, *d_blob = nullptr;
    size_t blob_bytes = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr;
    std::vector<cudaStream_t> branch;
    cudaEvent_t ev_fork = nullptr, ev_copied = nullptr;
    std::vector<cudaEvent_t> ev_join;
    bool copied_pending = false;
    unsigned char *d_codes = nullptr;  // decision codes of the requests' rows
    size_t codes_cap = 0;
    unsigned char *d_parts = nullptr;  // parts of the split requests' rows
    size_t parts_cap = 0;
};

namespace {

struct Req {
    int e;  // batch ensemble index
    const float *C;
    float *phi;
    int64_t n, ldc, ldp;
    size_t codes_off = 0;  // the request's region of the code arena
    int groups = 1;        // work items per tile (launch.h)
    size_t parts_off = 0;  // split: the request's region of the parts' scratch
};

// Classes are ensembles of one depth whose blocks of 32 rows fit an SM about equally often: a
// class's launch gives every block the shared memory of its widest ensemble, so a narrow one
// beside one of 300 features would run with half its warps.  64
// ensembles of 20 to 300 features, 2.05M rows: 19.3 ms with a class per depth, 16.5 so.
int class_room(const wdf_ensemble *e, const wdf::DevInfo &dev) {
    const int blocks = wdf::explain_blocks_per_sm(e->pk.D, e->pk.F, e->pk.quads, 32, dev);
    return blocks >= 7 ? 3 : blocks >= 5 ? 2 : blocks >= 3 ? 1 : 0;
}

bool tile_fits(const Cls &k, int tile_rows, const wdf::DevInfo &dev) {
    return (!k.wide || tile_rows == 32) && wdf::explain_fits(k.D, k.F_max, k.q_max, tile_rows, k.wide, dev);
}

void drop_graph(wdf_batch *b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
}

wdf_status wait_copied(wdf_batch *b) {
    if (b->copied_pending) WDF_CUDA(cudaEventSynchronize(b->ev_copied));
    b->copied_pending = false;
    return WDF_OK;
}

// Code arena regions of the requests (one per request, padded rows x the ensemble's code
// bytes per row), growing the arena if needed.  The regions' addresses travel in the
// blob, so the captured graph stays valid when the arena moves.
wdf_status place_codes(wdf_batch *b, std::vector<Req> *reqs) {
    size_t total = 0;
    for (Req &r : *reqs) {
        const wdf::Packed &p = b->ens[(size_t)r.e]->pk;
        r.codes_off = total;
        total += (size_t)padded_rows(r.n) / 32 * (size_t)p.quads * 16;
    }
    if (total > b->codes_cap) {
        wdf_status s = wait_copied(b);
        if (s != WDF_OK) return s;
        WDF_CUDA(cudaDeviceSynchronize());  // earlier launches may still read the old arena
        if (b->d_codes) cudaFree(b->d_codes);
        b->d_codes = nullptr;
        b->codes_cap = 0;
        const size_t cap = std::max<size_t>(total + total / 2, 1 << 20);
        WDF_CUDA(cudaMalloc((void **)&b->d_codes, cap));
        b->codes_cap = cap;
    }
    return WDF_OK;
}

// Splits the requests whose tiles would be the call's tail.  A tile walks all trees of its
// ensemble one after another (0.034 us per tree and leaf position, 2.2 ms for 257 trees of depth
// 8), and parts of the walk are independent; storing and adding parts costs a few percent, so a
// tile is cut into pieces of at most a quarter of the time that the whole call takes with
// every SM busy, as far as the scratch goes.  A call with many tiles is not split at all.
// Twelve ensembles, 87,079 rows in all: 2.45 -> 1.26 ms; a burst of 24 server requests 11.2 ->
// 10.5 ms; 163 tiles against 257 trees of depth 8 alone 2.3 -> 0.75 ms.
// tile_rows: of every class.
void plan_groups(const wdf_batch *b, const std::vector<int> &tile_rows, std::vector<Req> *reqs) {
    double call = 0.0;  // in tree leaves walked by one block at full occupancy
    for (const Req &r : *reqs) {
        const wdf::Packed &p = b->ens[(size_t)r.e]->pk;
        const Cls &k = b->cls[(size_t)b->cls_of[(size_t)r.e]];
        const int tc = tile_rows[(size_t)b->cls_of[(size_t)r.e]];
        call += (double)((r.n + tc - 1) / tc) * ((double)p.T * p.NL) /
                ((double)b->ctx->dev.sms * wdf::explain_blocks_per_sm(k.D, k.F_max, k.q_max, tc, b->ctx->dev));
    }
    size_t used = 0;
    for (Req &r : *reqs) {
        const wdf::Packed &p = b->ens[(size_t)r.e]->pk;
        const int P = wdf::explain_parts(p.T, p.D);
        const double want = std::ceil((double)p.T * p.NL / (0.25 * call));
        const size_t bytes = ((size_t)P * (size_t)r.n * (size_t)p.F * sizeof(float) + 255) & ~(size_t)255;
        r.groups = want >= P ? P : std::max(1, (int)want);
        if (r.n > (int64_t)(kPartsBytes / sizeof(float)) || used + bytes > kPartsBytes) r.groups = 1;
        if (r.groups > 1) {
            r.parts_off = used;
            used += bytes;
        }
    }
}

// Scratch for the planned parts, grown like the code arena.  Without memory for it the call
// runs with whole tiles.
wdf_status place_parts(wdf_batch *b, std::vector<Req> *reqs) {
    size_t total = 0;
    for (const Req &r : *reqs) {
        const wdf::Packed &p = b->ens[(size_t)r.e]->pk;
        if (r.groups > 1)
            total = r.parts_off + (size_t)wdf::explain_parts(p.T, p.D) * (size_t)r.n * (size_t)p.F * sizeof(float);
    }
    if (total > b->parts_cap) {
        wdf_status s = wait_copied(b);
        if (s != WDF_OK) return s;
        WDF_CUDA(cudaDeviceSynchronize());  // earlier launches may still use the old scratch
        if (b->d_parts) cudaFree(b->d_parts);
        b->d_parts = nullptr;
        b->parts_cap = 0;
        const size_t cap = std::min(std::max<size_t>(total + total / 2, 1 << 20), kPartsBytes);
        const cudaError_t e = cudaMalloc((void **)&b->d_parts, cap);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            b->d_parts = nullptr;
            for (Req &r : *reqs) r.groups = 1;
            return WDF_OK;
        }
        WDF_CUDA(e);
        b->parts_cap = cap;
    }
    return WDF_OK;
}

// Blob layout for the current capacities; reallocates (and drops the graph) if it grew.
wdf_status ensure_blob(wdf_batch *b, const std::vector<int> &need_reqs, const std::vector<int> &need_items,
                       const std::vector<int> &need_eitems, const std::vector<int> &need_tiles) {
    bool grow = b->h_blob == nullptr;
    for (size_t c = 0; c < b->cls.size(); ++c)
        if (need_reqs[c] > b->cls[c].cap_reqs || need_items[c] > b->cls[c].cap_items ||
            need_eitems[c] > b->cls[c].cap_eitems || need_tiles[c] > b->cls[c].cap_tiles)
            grow = true;
    if (!grow) return WDF_OK;
    wdf_status s = wait_copied(b);
    if (s != WDF_OK) return s;
    WDF_CUDA(cudaDeviceSynchronize());
    drop_graph(b);
    size_t off = 0;
    for (size_t c = 0; c < b->cls.size(); ++c) {
        Cls &k = b->cls[c];
        k.cap_reqs = std::max(k.cap_reqs, std::max(need_reqs[c], 4) * 3 / 2);
        k.cap_items = std::max(k.cap_items, std::max(need_items[c], 64) * 3 / 2);
        k.cap_eitems = std::max(k.cap_eitems, std::max(need_eitems[c], 64) * 3 / 2);
        k.cap_tiles = std::max(k.cap_tiles, std::max(need_tiles[c], 64) * 3 / 2);
        k.off_jobs = off;
        off = up16(off + k.members.size() * sizeof(wdf::ExplainJob));
        k.off_reqs = off;
        off = up16(off + (size_t)k.cap_reqs * sizeof(wdf::BatchRequest));
        k.off_items = off;
        off = up16(off + (size_t)k.cap_items * sizeof(int4));
        k.off_count = off;
        off = up16(off + (2 + (size_t)k.cap_tiles) * sizeof(int));
        k.off_eitems = off;
        off = up16(off + (size_t)k.cap_eitems * sizeof(int4));
        k.off_ecount = off;
        off = up16(off + sizeof(int));
    }
    if (b->h_blob) cudaFreeHost(b->h_blob);
    if (b->d_blob) cudaFree(b->d_blob);
    b->h_blob = nullptr;
    b->d_blob = nullptr;
    WDF_CUDA(cudaMallocHost((void **)&b->h_blob, off));
    WDF_CUDA(cudaMalloc((void **)&b->d_blob, off));
    std::memset(b->h_blob, 0, off);
    b->blob_bytes = off;
    return WDF_OK;
}

// 32-row blocks of an encode item: as few as give every resident block of an encode grid an
// item (an item reads its thresholds once, some 2 us, and takes 5 us a block), 16 at most.
int encode_item_blocks(const wdf_batch *b, const std::vector<Req> &reqs) {
    int64_t total = 0;
    for (const Req &r : reqs)
        total += padded_rows(r.n) / 32 * (int64_t)b->ens[(size_t)r.e]->pk.sgroup.size();
    const int64_t grid = 3 * (int64_t)b->ctx->dev.sms;
    return (int)std::max<int64_t>(1, std::min<int64_t>(kMostItemBlocks, (total + grid - 1) / grid));
}

// Writes one class's jobs, requests and items into the host blob.
int fill_class(wdf_batch *b, int c, const std::vector<Req> &reqs, int tile_rows) {
    Cls &k = b->cls[(size_t)c];
    auto *jobs = reinterpret_cast<wdf::ExplainJob *>(b->h_blob + k.off_jobs);
    for (size_t j = 0; j < k.members.size(); ++j) jobs[j] = b->ens[(size_t)k.members[j]]->job();
    auto *rq = reinterpret_cast<wdf::BatchRequest *>(b->h_blob + k.off_reqs);
    auto *items = reinterpret_cast<int4 *>(b->h_blob + k.off_items);
    auto *eitems = reinterpret_cast<int4 *>(b->h_blob + k.off_eitems);
    int nr = 0, ni = 0, ne = 0, nt = 0;
    const int eb = encode_item_blocks(b, reqs);
    for (const Req &r : reqs) {
        if (b->cls_of[(size_t)r.e] != c) continue;
        rq[nr] = wdf::BatchRequest{r.C,   r.phi, b->d_codes + r.codes_off, nullptr, r.n, r.ldc,
                                   r.ldp, b->slot_of[(size_t)r.e],  r.groups, nt};
        if (r.groups > 1) {
            rq[nr].parts = reinterpret_cast<float *>(b->d_parts + r.parts_off);
            nt += (int)((r.n + tile_rows - 1) / tile_rows);
        }
        for (int64_t c0 = 0; c0 < r.n; c0 += tile_rows)
            for (int g = 0; g < r.groups; ++g)
                items[ni++] = make_int4(b->slot_of[(size_t)r.e], nr, (int)(c0 >> 31) | g << wdf::kBatchGroupShift,
                                        (int)(c0 & 0x7FFFFFFF));
        const int64_t blocks = padded_rows(r.n) / 32;
        for (int64_t blk = 0; blk < blocks; blk += eb)
            for (int g = 0; g < (int)b->ens[(size_t)r.e]->pk.sgroup.size(); ++g)
                eitems[ne++] = make_int4(nr, g, (int)blk, (int)std::min<int64_t>(eb, blocks - blk));
        ++nr;
    }
    // longest first: blocks claim items in this order, so the cheap ones fill the tail of the
    // launch; then by ensemble and group, so that blocks at work together walk the same trees
    // (the folded vectors of 350 trees of depth 8 are three times the L2 cache: 56,000 rows 6.7
    // ms, with a tile's groups next to one another 8.1)
    auto cost = [&](const int4 &i) {
        return (double)b->ens[(size_t)k.members[(size_t)i.x]]->pk.T / rq[i.y].groups;
    };
    std::stable_sort(items, items + ni, [&](const int4 &a, const int4 &c) {
        const double ca = cost(a), cc = cost(c);
        if (ca != cc) return ca > cc;
        return a.x != c.x ? a.x < c.x : a.z >> wdf::kBatchGroupShift < c.z >> wdf::kBatchGroupShift;
    });
    int *hdr = reinterpret_cast<int *>(b->h_blob + k.off_count);
    hdr[0] = ni;  // item count
    std::memset(hdr + 1, 0, (1 + (size_t)nt) * sizeof(int));  // claim counter and tile counters, zero at every launch
    *reinterpret_cast<int *>(b->h_blob + k.off_ecount) = ne;
    return ni;
}

wdf_status capture(wdf_batch *b) {
    drop_graph(b);
    WDF_CUDA(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeRelaxed));
    cudaError_t e = cudaMemcpyAsync(b->d_blob, b->h_blob, b->blob_bytes, cudaMemcpyHostToDevice, b->cap);
    // an event-record node the host can wait on before rewriting the pinned blob
    if (e == cudaSuccess) e = cudaEventRecordWithFlags(b->ev_copied, b->cap, cudaEventRecordExternal);
    if (e == cudaSuccess) e = cudaEventRecord(b->ev_fork, b->cap);
    for (size_t c = 0; c < b->cls.size() && e == cudaSuccess; ++c) {
        const Cls &k = b->cls[c];
        e = cudaStreamWaitEvent(b->branch[c], b->ev_fork, 0);
        if (e == cudaSuccess)
            e = wdf::launch_encode_batch(reinterpret_cast<const wdf::ExplainJob *>(b->d_blob + k.off_jobs),
                                         reinterpret_cast<const wdf::BatchRequest *>(b->d_blob + k.off_reqs),
                                         reinterpret_cast<const int4 *>(b->d_blob + k.off_eitems),
                                         reinterpret_cast<const int *>(b->d_blob + k.off_ecount), k.thr_max, b->ctx->dev,
                                         b->branch[c]);
        if (e == cudaSuccess)
            e = wdf::launch_explain_batch(
                k.D, reinterpret_cast<const wdf::ExplainJob *>(b->d_blob + k.off_jobs),
                reinterpret_cast<const wdf::BatchRequest *>(b->d_blob + k.off_reqs),
                reinterpret_cast<const int4 *>(b->d_blob + k.off_items),
                reinterpret_cast<int *>(b->d_blob + k.off_count), k.F_max, k.q_max, k.tile_rows, k.wide, 0, b->ctx->dev,
                b->branch[c]);
        if (e == cudaSuccess) e = cudaEventRecord(b->ev_join[c], b->branch[c]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->cap, b->ev_join[c], 0);
    }
    cudaGraph_t g = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(b->cap, &g);
    wdf::count_launches(-2 * (int)b->cls.size());  // counted per graph launch instead
    if (e != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return fail(WDF_ECUDA, std::string("batch graph capture: ") + cudaGetErrorString(e));
    }
    if (e2 != cudaSuccess) return fail(WDF_ECUDA, std::string("cudaStreamEndCapture: ") + cudaGetErrorString(e2));
    b->graph = g;
    WDF_CUDA(cudaGraphInstantiate(&b->exec, b->graph, 0));
    return WDF_OK;
}

wdf_status gather_requests(wdf_batch *b, int32_t nreq, const int32_t *idx, const float *const *C, const int64_t *n,
                           const int64_t *ldc, float *const *phi, const int64_t *ldphi, std::vector<Req> *out) {
    if (nreq < 0 || (nreq > 0 && (!idx || !C || !n || !ldc || !phi || !ldphi)))
        return fail(WDF_EINVAL, "bad request arrays");
    out->clear();
    for (int i = 0; i < nreq; ++i) {
        if (idx[i] < 0 || idx[i] >= (int)b->ens.size()) return fail(WDF_EINVAL, "ensemble index out of range");
        const wdf_ensemble *e = b->ens[(size_t)idx[i]];
        if (!e->has_bg) return fail(WDF_EINVAL, "an ensemble of the batch has no background");
        if (n[i] < 0 || n[i] > wdf::kBatchMaxRows || (n[i] > 0 && (!C[i] || !phi[i])) || ldc[i] < e->pk.F || ldphi[i] < e->pk.F)
            return fail(WDF_EINVAL, "bad request " + std::to_string(i));
        if (n[i] > 0) out->push_back(Req{idx[i], C[i], phi[i], n[i], ldc[i], ldphi[i]});
    }
    return WDF_OK;
}

void count_needs(const wdf_batch *b, const std::vector<Req> &reqs, const std::vector<int> &tile_rows,
                 std::vector<int> *need_reqs, std::vector<int> *need_items, std::vector<int> *need_eitems,
                 std::vector<int> *need_tiles) {
    need_reqs->assign(b->cls.size(), 0);
    need_items->assign(b->cls.size(), 0);
    need_eitems->assign(b->cls.size(), 0);
    need_tiles->assign(b->cls.size(), 0);
    const int eb = encode_item_blocks(b, reqs);
    for (const Req &r : reqs) {
        const int c = b->cls_of[(size_t)r.e];
        (*need_reqs)[(size_t)c] += 1;
        const int tiles = (int)((r.n + tile_rows[(size_t)c] - 1) / tile_rows[(size_t)c]);
        (*need_items)[(size_t)c] += tiles * r.groups;
        (*need_tiles)[(size_t)c] += r.groups > 1 ? tiles : 0;
        (*need_eitems)[(size_t)c] +=
            (int)((padded_rows(r.n) / 32 + eb - 1) / eb) *
            (int)b->ens[(size_t)r.e]->pk.sgroup.size();
    }
}

}  // namespace

extern "C" {

wdf_status wdf_batch_create(wdf_ctx *ctx, int32_t n_ensembles, wdf_ensemble *const *ensembles, wdf_batch **out) {
    if (!ctx || !out || n_ensembles < 1 || !ensembles) return fail(WDF_EINVAL, "bad arguments");
    *out = nullptr;
    for (int i = 0; i < n_ensembles; ++i)
        if (!ensembles[i] || ensembles[i]->ctx != ctx) return fail(WDF_EINVAL, "ensemble missing or of another context");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != ctx->device) cudaSetDevice(ctx->device);
    wdf_batch *b = new wdf_batch();
    b->ctx = ctx_retain(ctx);
    b->ens.assign(ensembles, ensembles + n_ensembles);
    b->cls_of.assign((size_t)n_ensembles, -1);
    b->slot_of.assign((size_t)n_ensembles, -1);
    for (int i = 0; i < n_ensembles; ++i) {
        const int D = b->ens[(size_t)i]->pk.D, room = class_room(b->ens[(size_t)i], ctx->dev);
        int c = -1;
        const bool wide = b->ens[(size_t)i]->wide;
        for (size_t k = 0; k < b->cls.size(); ++k) {
            const Cls &o = b->cls[k];
            // its blocks hold the most features and the most codes of any member
            if (o.D == D && o.room == room && o.wide == wide &&
                wdf::explain_fits(D, std::max(o.F_max, b->ens[(size_t)i]->pk.F),
                                  std::max(o.q_max, b->ens[(size_t)i]->pk.quads), 32, wide, ctx->dev))
                c = (int)k;
        }
        if (c < 0) {
            b->cls.push_back(Cls());
            c = (int)b->cls.size() - 1;
            b->cls.back().D = D;
            b->cls.back().room = room;
            b->cls.back().wide = wide;
        }
        Cls &k = b->cls[(size_t)c];
        k.F_max = std::max(k.F_max, b->ens[(size_t)i]->pk.F);
        k.q_max = std::max(k.q_max, b->ens[(size_t)i]->pk.quads);
        k.thr_max = std::max(k.thr_max, b->ens[(size_t)i]->slices().max_group_thr);
        b->cls_of[(size_t)i] = c;
        b->slot_of[(size_t)i] = (int)k.members.size();
        k.members.push_back(i);
    }
    cudaError_t e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_copied, cudaEventDisableTiming);
    b->branch.assign(b->cls.size(), nullptr);
    b->ev_join.assign(b->cls.size(), nullptr);
    for (size_t c = 0; c < b->cls.size() && e == cudaSuccess; ++c) {
        Cls &k = b->cls[c];
        k.tile_rows = wdf::default_tile_rows(k.D, k.F_max, k.q_max, ctx->dev);
        if (!tile_fits(k, k.tile_rows, ctx->dev)) {
            e = cudaErrorInvalidConfiguration;
            break;
        }
        e = cudaStreamCreateWithFlags(&b->branch[c], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_join[c], cudaEventDisableTiming);
    }
    if (prev >= 0 && prev != ctx->device) cudaSetDevice(prev);
    if (e != cudaSuccess) {
        wdf_batch_destroy(b);
        return fail(WDF_ECUDA, std::string("wdf_batch_create: ") + cudaGetErrorString(e));
    }
    *out = b;
    return WDF_OK;
}

void wdf_batch_destroy(wdf_batch *b) {
    if (!b) return;
    int prev = -1;
    cudaGetDevice(&prev);
    if (b->ctx && prev != b->ctx->device) cudaSetDevice(b->ctx->device);
    cudaDeviceSynchronize();
    drop_graph(b);
    if (b->h_blob) cudaFreeHost(b->h_blob);
    if (b->d_blob) cudaFree(b->d_blob);
    if (b->d_codes) cudaFree(b->d_codes);
    if (b->d_parts) cudaFree(b->d_parts);
    for (cudaStream_t s : b->branch)
        if (s) cudaStreamDestroy(s);
    for (cudaEvent_t ev : b->ev_join)
        if (ev) cudaEventDestroy(ev);
    if (b->cap) cudaStreamDestroy(b->cap);
    if (b->ev_fork) cudaEventDestroy(b->ev_fork);
    if (b->ev_copied) cudaEventDestroy(b->ev_copied);
    if (b->ctx && prev >= 0 && prev != b->ctx->device) cudaSetDevice(prev);
    ctx_release(b->ctx);
    delete b;
}

wdf_status wdf_batch_explain(wdf_batch *b, int32_t n_requests, const int32_t *ensemble_index, const float *const *C,
                             const int64_t *n, const int64_t *ldc, float *const *phi, const int64_t *ldphi,
                             void *stream) {
    wdf::TraceRange trace_("wdf_batch_explain");
    if (!b) return fail(WDF_EINVAL, "batch is null");
    std::vector<Req> reqs;
    wdf_status s = gather_requests(b, n_requests, ensemble_index, C, n, ldc, phi, ldphi, &reqs);
    if (s != WDF_OK) return s;
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != b->ctx->device) cudaSetDevice(b->ctx->device);
    std::vector<int> tiles, need_reqs, need_items, need_eitems, need_tiles;
    for (const Cls &k : b->cls) tiles.push_back(k.tile_rows);
    plan_groups(b, tiles, &reqs);
    count_needs(b, reqs, tiles, &need_reqs, &need_items, &need_eitems, &need_tiles);
    s = ensure_blob(b, need_reqs, need_items, need_eitems, need_tiles);
    if (s == WDF_OK) s = place_codes(b, &reqs);
    if (s == WDF_OK) s = place_parts(b, &reqs);
    if (s == WDF_OK) s = wait_copied(b);
    if (s == WDF_OK) {
        for (size_t c = 0; c < b->cls.size(); ++c) fill_class(b, (int)c, reqs, b->cls[c].tile_rows);
        if (!b->exec) s = capture(b);
    }
    if (s == WDF_OK) {
        const cudaError_t e = cudaGraphLaunch(b->exec, (cudaStream_t)stream);
        if (e != cudaSuccess) s = fail(WDF_ECUDA, std::string("cudaGraphLaunch: ") + cudaGetErrorString(e));
        else {
            b->copied_pending = true;
            wdf::count_launches(2 * (int)b->cls.size());
        }
    }
    if (prev >= 0 && prev != b->ctx->device) cudaSetDevice(prev);
    return s;
}

wdf_status wdf_batch_autotune(wdf_batch *b, int32_t n_requests, const int32_t *ensemble_index, const float *const *C,
                              const int64_t *n, const int64_t *ldc, float *const *phi, const int64_t *ldphi,
                              int32_t reps, const char *cache_path, void *stream) {
    wdf::TraceRange trace_("wdf_batch_autotune");
    if (!b) return fail(WDF_EINVAL, "batch is null");
    std::vector<Req> reqs;
    wdf_status s = gather_requests(b, n_requests, ensemble_index, C, n, ldc, phi, ldphi, &reqs);
    if (s != WDF_OK) return s;
    reps = std::max(1, reps);
    // cached choices: "depth features_rounded code_bytes_rounded tile_rows ms" per line
    std::vector<std::vector<int>> cached;
    if (cache_path) {
        std::ifstream in(cache_path);
        std::string line;
        while (std::getline(in, line)) {
            std::istringstream ls(line);
            int d, f, x, t;
            if (ls >> d >> f >> x >> t) cached.push_back({d, f, x, t});
        }
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != b->ctx->device) cudaSetDevice(b->ctx->device);
    cudaStream_t st = (cudaStream_t)stream;
    const int cand[3] = {32, 64, 128};
    // tile_rows 32 and every part an item needs the most
    std::vector<int> t32(b->cls.size(), 32), need_reqs, need_items, need_eitems, need_tiles;
    for (Req &r : reqs) r.groups = wdf::explain_parts(b->ens[(size_t)r.e]->pk.T, b->ens[(size_t)r.e]->pk.D);
    count_needs(b, reqs, t32, &need_reqs, &need_items, &need_eitems, &need_tiles);
    s = ensure_blob(b, need_reqs, need_items, need_eitems, need_tiles);
    if (s == WDF_OK) s = place_codes(b, &reqs);
    if (s == WDF_OK) s = wait_copied(b);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (s == WDF_OK && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
        s = fail(WDF_ECUDA, "cudaEventCreate");
    std::ofstream log;
    if (s == WDF_OK && cache_path) log.open(cache_path, std::ios::app);
    for (size_t c = 0; c < b->cls.size() && s == WDF_OK; ++c) {
        Cls &k = b->cls[c];
        if (need_reqs[c] == 0) continue;
        const int fkey = (k.F_max + 31) / 32 * 32, xkey = (k.q_max / 2 + 31) / 32 * 32;  // half a byte per quad and row
        int hit = 0;
        for (const auto &row : cached)
            if (row[0] == k.D && row[1] == fkey && row[2] == xkey && (row[3] == 32 || row[3] == 64 || row[3] == 128) &&
                tile_fits(k, row[3], b->ctx->dev))
                hit = row[3];
        if (hit) {
            k.tile_rows = hit;
            continue;
        }
        float best_ms = 1e30f;
        int best = k.tile_rows;
        // the rows' codes do not depend on the tile size: encode them once
        for (Req &r : reqs) r.groups = 1;
        fill_class(b, (int)c, reqs, k.tile_rows);
        {
            cudaError_t e = cudaMemcpyAsync(b->d_blob, b->h_blob, b->blob_bytes, cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess)
                e = wdf::launch_encode_batch(reinterpret_cast<const wdf::ExplainJob *>(b->d_blob + k.off_jobs),
                                             reinterpret_cast<const wdf::BatchRequest *>(b->d_blob + k.off_reqs),
                                             reinterpret_cast<const int4 *>(b->d_blob + k.off_eitems),
                                             reinterpret_cast<const int *>(b->d_blob + k.off_ecount), k.thr_max,
                                             b->ctx->dev, st);
            if (e != cudaSuccess) {
                s = fail(WDF_ECUDA, std::string("autotune: ") + cudaGetErrorString(e));
                break;
            }
        }
        for (int tc : cand) {
            if (!tile_fits(k, tc, b->ctx->dev)) continue;
            std::vector<int> tiles;
            for (const Cls &o : b->cls) tiles.push_back(&o == &k ? tc : o.tile_rows);
            plan_groups(b, tiles, &reqs);
            s = place_parts(b, &reqs);
            if (s != WDF_OK) break;
            fill_class(b, (int)c, reqs, tc);
            cudaError_t e = cudaMemcpyAsync(b->d_blob, b->h_blob, b->blob_bytes, cudaMemcpyHostToDevice, st);
            float ms = 0.0f;
            for (int r = -1; r < reps && e == cudaSuccess; ++r) {  // r = -1 warms up
                if (r == 0) e = cudaEventRecord(e0, st);
                if (e == cudaSuccess)  // reset the claim and tile counters of this class
                    e = cudaMemsetAsync(b->d_blob + k.off_count + sizeof(int), 0, (1 + (size_t)k.cap_tiles) * sizeof(int),
                                        st);
                if (e == cudaSuccess)
                    e = wdf::launch_explain_batch(k.D, reinterpret_cast<const wdf::ExplainJob *>(b->d_blob + k.off_jobs),
                                                  reinterpret_cast<const wdf::BatchRequest *>(b->d_blob + k.off_reqs),
                                                  reinterpret_cast<const int4 *>(b->d_blob + k.off_items),
                                                  reinterpret_cast<int *>(b->d_blob + k.off_count), k.F_max, k.q_max, tc,
                                                  k.wide, 0, b->ctx->dev, st);
            }
            if (e == cudaSuccess) e = cudaEventRecord(e1, st);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e != cudaSuccess) {
                s = fail(WDF_ECUDA, std::string("autotune: ") + cudaGetErrorString(e));
                break;
            }
            ms /= (float)reps;
            if (ms < best_ms) {
                best_ms = ms;
                best = tc;
            }
        }
        if (s != WDF_OK) break;
        k.tile_rows = best;
        if (log.is_open()) log << k.D << " " << fkey << " " << xkey << " " << best << " " << best_ms << "\n";
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    drop_graph(b);  // recaptured with the chosen tile sizes on the next explain
    if (prev >= 0 && prev != b->ctx->device) cudaSetDevice(prev);
    return s;
}

wdf_status wdf_batch_tile_rows(const wdf_batch *b, int32_t depth, int32_t *tile_rows) {
    if (!b || !tile_rows) return fail(WDF_EINVAL, "null argument");
    *tile_rows = -1;
    for (const Cls &k : b->cls)
        if (k.D == depth && (*tile_rows < 0 || k.tile_rows < *tile_rows)) *tile_rows = k.tile_rows;
    return WDF_OK;
}

}  // extern "C"
