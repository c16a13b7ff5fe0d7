// Depth and tile dispatch of the consumer kernels (k_explain.cuh); the kernels are
// compiled in the k_explain_d*.cu translation units.
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "k_explain.cuh"

namespace wdf {

namespace {
std::mutex g_tmu;
bool g_timing = false;
std::vector<std::pair<cudaEvent_t, cudaEvent_t>> g_tev;

void drop_events() {
    for (auto &p : g_tev) {
        cudaEventDestroy(p.first);
        cudaEventDestroy(p.second);
    }
    g_tev.clear();
}
}  // namespace

void explain_timing(bool on) {
    std::lock_guard<std::mutex> lk(g_tmu);
    drop_events();
    g_timing = on;
}

cudaError_t explain_timing_read(double *ms, int64_t *launches) {
    std::lock_guard<std::mutex> lk(g_tmu);
    double total = 0.0;
    cudaError_t err = cudaSuccess;
    for (auto &p : g_tev) {
        float t = 0.0f;
        if (err == cudaSuccess) err = cudaEventSynchronize(p.second);
        if (err == cudaSuccess) err = cudaEventElapsedTime(&t, p.first, p.second);
        total += t;
    }
    *ms = total;
    *launches = (int64_t)g_tev.size();
    drop_events();
    return err;
}

WDF_EXPLAIN_DEPTH(2, extern)
WDF_EXPLAIN_DEPTH(3, extern)
WDF_EXPLAIN_DEPTH(4, extern)
WDF_EXPLAIN_DEPTH(5, extern)
WDF_EXPLAIN_DEPTH(6, extern)
WDF_EXPLAIN_DEPTH(7, extern)
WDF_EXPLAIN_DEPTH(8, extern)

template <int D>
static cudaError_t explain_depth(const unsigned char *codes, int64_t n, const ExplainJob &job, float *phi,
                                 int64_t ldp, int tile_rows, const DevInfo &dev, cudaStream_t st) {
    switch (tile_rows) {
        case 32: return explain_t<D, 32>(codes, n, job, phi, ldp, dev, st);
        case 128: return explain_t<D, 128>(codes, n, job, phi, ldp, dev, st);
        default: return explain_t<D, 64>(codes, n, job, phi, ldp, dev, st);
    }
}

template <int D>
static cudaError_t batch_depth(const ExplainJob *jobs, const BatchRequest *reqs, const int4 *items, int *n_items,
                               int F_max, int q_max, int tile_rows, int grid, const DevInfo &dev, cudaStream_t st) {
    switch (tile_rows) {
        case 32: return batch_t<D, 32>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
        case 128: return batch_t<D, 128>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
        default: return batch_t<D, 64>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
    }
}

// The tile that keeps most warps on an SM; 32 rows where 64 keep no more (the same speed at
// depth 6 and 127 features, 545-560 SM clocks per warp and tree; 3-7 % faster for deeper trees
// and 20 % at 255 features, whose smaller blocks fill the shared memory better).
int default_tile_rows(int D, int F, int quads, const DevInfo &dev) {
    int best = 32;
    size_t most = 0;
    for (int tc : {32, 64}) {
        const size_t smem = explain_smem_bytes(D, F, quads, tc);
        if (smem > dev.smem_optin) continue;
        const size_t warps = std::min<size_t>(explain_warps(D), (dev.smem_optin + 1024) / (smem + 1024) * (tc / 16));
        if (warps > most) {
            most = warps;
            best = tc;
        }
    }
    return best;
}

// Rows per encoded chunk: the decision codes of a chunk live in a stream-ordered
// scratch allocation (so concurrent calls on other streams never share it).
constexpr int64_t kExplainChunkRows = 1 << 20;

cudaError_t launch_explain(int D, const float *C, int64_t n, int64_t ldc, const ExplainJob &job, float *phi,
                           int64_t ldp, int tile_rows, const DevInfo &dev, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (D < 2 || D > 8) return cudaErrorInvalidValue;
    if (tile_rows <= 0) tile_rows = default_tile_rows(D, job.F, job.sa.quads, dev);
    const int64_t chunk = std::min(n, kExplainChunkRows);
    const int64_t pad = 128;  // every tile size divides it
    unsigned char *codes = nullptr;
    cudaError_t err = cudaMallocAsync(reinterpret_cast<void **>(&codes), (size_t)((chunk + pad - 1) / pad * pad) / 32 * job.sa.quads * 16, st);
    if (err != cudaSuccess) return err;
    for (int64_t r0 = 0; r0 < n && err == cudaSuccess; r0 += chunk) {
        const int64_t rows = std::min(chunk, n - r0);
        err = launch_encode_slices(C + r0 * ldc, rows, ldc, job.sa, (rows + pad - 1) / pad * pad, codes, dev, st);
        if (err != cudaSuccess) break;
        float *out = phi + r0 * ldp;
        cudaEvent_t ev0 = nullptr, ev1 = nullptr;
        {
            std::lock_guard<std::mutex> lk(g_tmu);
            if (g_timing && cudaEventCreate(&ev0) == cudaSuccess) {
                if (cudaEventCreate(&ev1) == cudaSuccess) {
                    cudaEventRecord(ev0, st);
                } else {
                    cudaEventDestroy(ev0);
                    ev0 = ev1 = nullptr;
                }
            }
        }
        switch (D) {
            case 2: err = explain_depth<2>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
            case 3: err = explain_depth<3>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
            case 4: err = explain_depth<4>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
            case 5: err = explain_depth<5>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
            case 6: err = explain_depth<6>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
            case 7: err = explain_depth<7>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
            default: err = explain_depth<8>(codes, rows, job, out, ldp, tile_rows, dev, st); break;
        }
        if (ev1) {  // the pair is kept only once both ends are recorded
            std::lock_guard<std::mutex> lk(g_tmu);
            cudaEventRecord(ev1, st);
            g_tev.emplace_back(ev0, ev1);
        }
    }
    const cudaError_t ferr = cudaFreeAsync(codes, st);
    return err != cudaSuccess ? err : ferr;
}

cudaError_t launch_explain_batch(int D, const ExplainJob *jobs, const BatchRequest *reqs, const int4 *items,
                                 int *n_items, int F_max, int q_max, int tile_rows, int grid, const DevInfo &dev,
                                 cudaStream_t st) {
    switch (D) {
        case 2: return batch_depth<2>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        case 3: return batch_depth<3>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        case 4: return batch_depth<4>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        case 5: return batch_depth<5>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        case 6: return batch_depth<6>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        case 7: return batch_depth<7>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        case 8: return batch_depth<8>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, grid, dev, st);
        default: return cudaErrorInvalidValue;
    }
}

// One block per (tree, image).
__global__ void k_images(int D, int T, const UnitNode *__restrict__ unit, const TreeMeta *__restrict__ meta,
                         const int32_t *__restrict__ flfeat, const uint8_t *__restrict__ flrep,
                         unsigned char *__restrict__ image) {
    const int t = blockIdx.x, i = blockIdx.y, tid = threadIdx.x;
    unsigned char *dst = image + ((size_t)i * T + t) * image_bytes(D);
    const int nu = units_per_tree(D) * 32, fl = flush_len(D), xs = image_rows(i) + 1;
    for (int k = tid; k < nu; k += blockDim.x) reinterpret_cast<UnitNode *>(dst)[k] = unit[(size_t)t * nu + k];
    if (tid < 4) {
        const TreeMeta &m = meta[t];
        reinterpret_cast<uint64_t *>(dst + image_flags(D))[tid] =
            tid == 0 ? m.live : tid == 1 ? m.flush : tid == 2 ? m.real : 0ull;
    }
    for (int k = tid; k < fl; k += blockDim.x)
        reinterpret_cast<uint16_t *>(dst + image_offsets(D))[k] = (uint16_t)(flfeat[(size_t)t * fl + k] * xs);
    for (int k = tid; k < fl / 8; k += blockDim.x) dst[image_repeats(D) + k] = flrep[(size_t)t * (fl / 8) + k];
}

cudaError_t launch_images(int D, int T, const UnitNode *unit, const TreeMeta *meta, const int32_t *flfeat,
                          const uint8_t *flrep, unsigned char *image, cudaStream_t st) {
    k_images<<<dim3((unsigned)T, kImages), 128, 0, st>>>(D, T, unit, meta, flfeat, flrep, image);
    count_launches(1);
    return cudaGetLastError();
}

size_t explain_smem_bytes(int D, int F, int quads, int tile_rows) {
    switch (D * 1000 + tile_rows) {
#define WDF_SMEM_CASE(d, tc) \
    case d * 1000 + tc: return ExLayout<d>(F, quads, tc).total;
        WDF_SMEM_CASE(2, 32) WDF_SMEM_CASE(2, 64) WDF_SMEM_CASE(2, 128)
        WDF_SMEM_CASE(3, 32) WDF_SMEM_CASE(3, 64) WDF_SMEM_CASE(3, 128)
        WDF_SMEM_CASE(4, 32) WDF_SMEM_CASE(4, 64) WDF_SMEM_CASE(4, 128)
        WDF_SMEM_CASE(5, 32) WDF_SMEM_CASE(5, 64) WDF_SMEM_CASE(5, 128)
        WDF_SMEM_CASE(6, 32) WDF_SMEM_CASE(6, 64) WDF_SMEM_CASE(6, 128)
        WDF_SMEM_CASE(7, 32) WDF_SMEM_CASE(7, 64) WDF_SMEM_CASE(7, 128)
        WDF_SMEM_CASE(8, 32) WDF_SMEM_CASE(8, 64) WDF_SMEM_CASE(8, 128)
#undef WDF_SMEM_CASE
        default: return (size_t)-1;
    }
}

}  // namespace wdf
