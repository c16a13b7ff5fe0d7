// Depth and tile dispatch of the consumer kernels (k_explain.cuh); the kernels are
// compiled in the k_explain_d*.cu translation units.
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "explain_plan.h"
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
WDF_EXPLAIN_WIDE(2, extern)
WDF_EXPLAIN_WIDE(3, extern)
WDF_EXPLAIN_WIDE(4, extern)
WDF_EXPLAIN_WIDE(5, extern)
WDF_EXPLAIN_WIDE(6, extern)
WDF_EXPLAIN_WIDE(7, extern)
WDF_EXPLAIN_WIDE(8, extern)

template <int D>
static cudaError_t explain_depth(const unsigned char *codes, int64_t n, const ExplainJob &job, float *phi,
                                 int64_t ldp, int tile_rows, int splits, float *scratch, const DevInfo &dev,
                                 cudaStream_t st) {
    if (job.wide) return explain_t<D, 32, true>(codes, n, job, phi, ldp, splits, scratch, dev, st);
    switch (tile_rows) {
        case 32: return explain_t<D, 32, false>(codes, n, job, phi, ldp, splits, scratch, dev, st);
        case 128: return explain_t<D, 128, false>(codes, n, job, phi, ldp, splits, scratch, dev, st);
        default: return explain_t<D, 64, false>(codes, n, job, phi, ldp, splits, scratch, dev, st);
    }
}

template <int D>
static cudaError_t batch_depth(const ExplainJob *jobs, const BatchRequest *reqs, const int4 *items, int *n_items,
                               int F_max, int q_max, int tile_rows, bool wide, int grid, const DevInfo &dev,
                               cudaStream_t st) {
    if (wide) return batch_t<D, 32, true>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
    switch (tile_rows) {
        case 32: return batch_t<D, 32, false>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
        case 128: return batch_t<D, 128, false>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
        default: return batch_t<D, 64, false>(jobs, reqs, items, n_items, F_max, q_max, grid, dev, st);
    }
}

int explain_blocks_per_sm(int D, int F, int quads, int tile_rows, const DevInfo &dev) {
    const size_t smem = explain_smem_bytes(D, F, quads, tile_rows);
    const size_t room = explain_carveout(D, tile_rows, smem) ? kExplainCarveout : dev.smem_optin + 1024;
    return std::max(1, std::min((int)(room / (smem + 1024)), kExplainWarps * 16 / tile_rows));
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
        const size_t warps = std::min<size_t>(kExplainWarps, (dev.smem_optin + 1024) / (smem + 1024) * (tc / 16));
        if (warps > most) {
            most = warps;
            best = tc;
        }
    }
    return best;
}

// phi = the parts' sums, added in part order; one thread per element of a row.
__global__ void k_add_parts(const float *__restrict__ scratch, int P, int64_t n, int F, float *__restrict__ phi,
                            int64_t ldp) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * F) return;
    float x = __ldg(scratch + i);
    for (int p = 1; p < P; ++p) x += __ldg(scratch + (size_t)p * n * F + i);
    phi[i / F * ldp + i % F] = x;
}

// phi from the node values of k_values: a warp adds one feature's nodes of one part and 32 rows in
// their order, then a thread adds the parts in theirs.  part_warps (a power of two, at most
// kSumWarps) warps per feature, so that a large ensemble's parts are summed side by side; the
// node list is read 32 entries at a time and the values 16 at a time, so their latency
// overlaps; only the additions are a chain.  777 rows, 500 trees of depth 7 and 112 features, the
// whole call: 122 us with a warp per feature for all parts, 88 so.
constexpr int kSumWarps = 8;
__global__ void __launch_bounds__(32 * kSumWarps) k_sum_values(const float *__restrict__ values, int FL,
                                                              const int32_t *__restrict__ vlist,
                                                              const int32_t *__restrict__ voff, int T, int F, int P,
                                                              int part_warps, int64_t n, float *__restrict__ phi,
                                                              int64_t ldp) {
    __shared__ float out[32][kSumWarps + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, here = kSumWarps / part_warps;  // features of a block
    const int f = blockIdx.x * here + warp / part_warps, p = warp % part_warps;
    const float *v = values + (size_t)blockIdx.y * T * FL * 32 + lane;
    const bool on = f < F && p < P;
    const int off = on && lane < 2 ? __ldg(voff + (size_t)f * P + p + lane) : 0;
    const int beg = __shfl_sync(0xFFFFFFFFu, off, 0), end = __shfl_sync(0xFFFFFFFFu, off, 1);
    int mine = beg + lane < end ? __ldg(vlist + beg + lane) : 0;
    previous_done();  // the node values
    float acc = 0.0f;
    for (int k0 = beg; k0 < end; k0 += 32) {
        const int cnt = min(32, end - k0), ahead = k0 + 32 + lane;
        const int next = ahead < end ? __ldg(vlist + ahead) : 0;
#pragma unroll
        for (int h = 0; h < 32; h += 16) {
            float x[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int i = __shfl_sync(0xFFFFFFFFu, mine, h + k);
                x[k] = h + k < cnt ? v[(size_t)i * 32] : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (h + k < cnt) acc += x[k];
        }
        mine = next;
    }
    out[lane][warp] = acc;
    __syncthreads();
    const int r = threadIdx.x / kSumWarps, c = threadIdx.x % kSumWarps, fc = blockIdx.x * here + c;
    const int64_t row = (int64_t)blockIdx.y * 32 + r;
    if (c < here && row < n && fc < F) {
        float total = out[r][c * part_warps];
        for (int k = 1; k < P; ++k) total += out[r][c * part_warps + k];
        phi[row * ldp + fc] = total;
    }
}

template <int D>
static cudaError_t explain_values(const unsigned char *codes, int64_t n, const ExplainJob &job, float *phi, int64_t ldp,
                                  float *values, const DevInfo &dev, cudaStream_t st) {
    cudaError_t err = values_t<D>(codes, n, job, values, dev, st);
    if (err != cudaSuccess) return err;
    const int P = explain_parts(job.T, D);
    int part_warps = 1;
    while (part_warps < P) part_warps *= 2;
    static_assert(kSumWarps >= 8, "a warp per part");
    const int here = kSumWarps / part_warps;
    const dim3 grid((unsigned)((job.F + here - 1) / here), (unsigned)((n + 31) / 32));
    err = launch_dependent(k_sum_values, grid, 32 * kSumWarps, 0, st, (const float *)values, flush_len(D), job.vlist,
                           job.voff, job.T, job.F, P, part_warps, n, phi, ldp);
    count_launches(1);
    return err != cudaSuccess ? err : cudaGetLastError();
}

// Rows per encoded chunk: the decision codes of a chunk live in a stream-ordered
// scratch allocation (so concurrent calls on other streams never share it).
constexpr int64_t kExplainChunkRows = 1 << 20;

cudaError_t launch_explain(int D, const float *C, int64_t n, int64_t ldc, const ExplainJob &job, float *phi,
                           int64_t ldp, int tile_rows, const DevInfo &dev, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (D < 2 || D > 8) return cudaErrorInvalidValue;
    if (job.wide) tile_rows = 32;
    if (tile_rows <= 0) tile_rows = default_tile_rows(D, job.F, job.sa.quads, dev);
    if (explain_smem_bytes(D, job.F, job.sa.quads, tile_rows, job.wide) > dev.smem_optin)
        return cudaErrorInvalidConfiguration;
    const int64_t chunk = std::min(n, kExplainChunkRows);
    const int64_t pad = 128;  // every tile size divides it
    const size_t code_bytes = (size_t)((chunk + pad - 1) / pad * pad) / 32 * job.sa.quads * 16;
    ExplainPlan plan = explain_plan(D, chunk, job.T, job.F, tile_rows, dev.sms,
                                    explain_blocks_per_sm(D, job.F, job.sa.quads, tile_rows, dev),
                                    (size_t)job.sa.quads * 16 <= dev.smem_optin);
    unsigned char *codes = nullptr;
    cudaError_t err = take_scratch(&plan, chunk, code_bytes, cudaErrorMemoryAllocation, [&](size_t bytes) {
        const cudaError_t e = cudaMallocFromPoolAsync(reinterpret_cast<void **>(&codes), bytes, dev.pool, st);
        if (e == cudaErrorMemoryAllocation) cudaGetLastError();  // reported by its return value alone
        return e;
    });
    if (err != cudaSuccess) return err;
    const int splits = plan.splits;
    float *scratch = plan.scratch_floats ? reinterpret_cast<float *>(codes + scratch_at(code_bytes)) : nullptr;
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
        for (int64_t q0 = 0; q0 < rows && err == cudaSuccess; q0 += plan.rows) {
            const int64_t here = std::min(plan.rows, rows - q0);
            const unsigned char *block = codes + (size_t)(q0 / 32) * job.sa.quads * 16;
            float *to = out + q0 * ldp;
            switch (D) {
#define WDF_EXPLAIN_CASE(d)                                                                                     \
    case d:                                                                                                     \
        err = splits == 0 ? explain_values<d>(block, here, job, to, ldp, scratch, dev, st)                      \
                          : explain_depth<d>(block, here, job, to, ldp, tile_rows, splits, scratch, dev, st);   \
        break;
                WDF_EXPLAIN_CASE(2) WDF_EXPLAIN_CASE(3) WDF_EXPLAIN_CASE(4) WDF_EXPLAIN_CASE(5)
                WDF_EXPLAIN_CASE(6) WDF_EXPLAIN_CASE(7) WDF_EXPLAIN_CASE(8)
#undef WDF_EXPLAIN_CASE
            }
            if (err == cudaSuccess && splits > 1) {
                k_add_parts<<<(unsigned)((here * job.F + 255) / 256), 256, 0, st>>>(
                    scratch, explain_parts(job.T, D), here, job.F, to, ldp);
                count_launches(1);
                err = cudaGetLastError();
            }
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
                                 int *n_items, int F_max, int q_max, int tile_rows, bool wide, int grid,
                                 const DevInfo &dev, cudaStream_t st) {
    switch (D) {
        case 2: return batch_depth<2>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        case 3: return batch_depth<3>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        case 4: return batch_depth<4>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        case 5: return batch_depth<5>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        case 6: return batch_depth<6>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        case 7: return batch_depth<7>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        case 8: return batch_depth<8>(jobs, reqs, items, n_items, F_max, q_max, tile_rows, wide, grid, dev, st);
        default: return cudaErrorInvalidValue;
    }
}

// One block per (tree, image).  wide: the one image of an ensemble of wide tiles.
__global__ void k_images(int D, int T, bool wide, const UnitNode *__restrict__ unit, const TreeMeta *__restrict__ meta,
                         const int32_t *__restrict__ flfeat, const uint8_t *__restrict__ flrep,
                         unsigned char *__restrict__ image) {
    const int t = blockIdx.x, i = blockIdx.y, tid = threadIdx.x, nt = blockDim.x, xs = wide ? 32 : image_rows(i) + 1;
    const int UPT = units_per_tree(D), CU = chunk_units(D), GS = gather_group(D), GB = flush_group_len(D) / 8;
    const int CP = chunk_positions(D);
    unsigned char *dst = image + ((size_t)i * T + t) * image_bytes(D);
    const UnitNode *src = unit + (size_t)t * UPT * 32;
    const int32_t *feat = flfeat + (size_t)t * flush_len(D);
    const uint8_t *rep = flrep + (size_t)t * flush_batches(D);
    const TreeMeta &m = meta[t];
    for (int c = 0; c < tree_chunks(D); ++c, dst += chunk_bytes(D)) {
        // batch b of the chunk is batch at(b) of the tree
        auto at = [&](int b) { return b < CU * GB ? c * CU * GB + b : UPT * GB; };
        for (int k = tid; k < 32 * CU; k += nt) reinterpret_cast<UnitNode *>(dst)[k] = src[c * CU * 32 + k];
        for (int k = tid; k < CP; k += nt)
            reinterpret_cast<uint16_t *>(dst + chunk_offsets(D))[k] = (uint16_t)(feat[8 * at(k / 8) + k % 8] * xs);
        for (int k = chunk_repeats(D) + tid; k < chunk_bytes(D); k += nt) {
            const int b = k - chunk_repeats(D);
            dst[k] = b < CP / 8 ? rep[at(b)] : 0;
        }
        if (tid < CU) {
            const int u = c * CU + tid, nb = GB + (UPT > 1 ? 1 : 0);
            uint32_t f = (uint32_t)(m.live >> (u * GS)) & ((1u << GS) - 1u);
            for (int b = 0; b < nb; ++b) {
                const int tb = b < GB ? u * GB + b : UPT * GB;
                f |= (uint32_t)((m.flush >> tb) & 1u) << (8 + b) | (uint32_t)((m.real >> tb) & 1u) << (16 + b);
            }
            reinterpret_cast<uint32_t *>(dst + chunk_flags(D))[tid] = f;
        }
    }
    if (unit_top(D) > 1 && tid < 8)  // lane 31 of unit u is node u
        reinterpret_cast<UnitNode *>(dst)[tid] = src[(tid < UPT ? tid : 0) * 32 + 31];
}

cudaError_t launch_images(int D, int T, bool wide, const UnitNode *unit, const TreeMeta *meta, const int32_t *flfeat,
                          const uint8_t *flrep, unsigned char *image, cudaStream_t st) {
    k_images<<<dim3((unsigned)T, (unsigned)(wide ? 1 : kImages)), 128, 0, st>>>(D, T, wide, unit, meta, flfeat, flrep, image);
    count_launches(1);
    return cudaGetLastError();
}

size_t explain_smem_bytes(int D, int F, int quads, int tile_rows, bool wide) {
    switch (D * 1000 + tile_rows) {
#define WDF_SMEM_CASE(d, tc) \
    case d * 1000 + tc: return ExLayout<d>(F, quads, tc, wide && tc == 32).total;
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
