// Decision codes (tree_layout.h) of consumer and background rows.
#include <algorithm>

#include "launch.h"
#include "wdf_device.cuh"

namespace wdf {

// A block keeps the search trees of one group of packs in
// shared memory and walks 32-row blocks: the rows' values are read along the rows (the
// next block's while this one is searched), then a warp takes a pack of eight columns, lane
// = row: eight searches side by side (one shared load, compare and add per level; siblings
// of a level lie side by side, so lanes at different nodes of the first five levels read
// different banks), four bits of the eight codes packed into one word per lane, and a
// 32 x 32 bit transpose gives the pack's eight quads, written as 128 contiguous bytes.
// Issue-bound (76 %): 0.36 ms per 1M rows of 127 columns, where a byte per code and a search
// per (row, column) in global memory took 0.58 ms.
constexpr int kSliceThreads = 256, kSliceWarps = kSliceThreads / 32;
constexpr int kSliceCols = 8 * kSliceGroupPacks, kSliceXs = kSliceCols + 1;
constexpr int kSliceRows = 32 / kSliceWarps, kSliceRuns = kSliceCols / 32;

size_t slice_smem(int max_group_thr) { return ((size_t)32 * kSliceXs + 32 + (size_t)max_group_thr) * 4; }

// The codes of group g's columns for 32-row blocks b0, b0 + step, ... below b1 of rows
// [0, rows) of X.  All threads of the block call it.
__device__ __forceinline__ void encode_group(const float *__restrict__ X, int64_t rows, int64_t ldx,
                                             const SliceArrays &sa, int group, int64_t b0, int64_t b1, int64_t step,
                                             unsigned char *__restrict__ codes, float *smem) {
    float *xs = smem, *st = smem + 32 * kSliceXs + 32;  // 16-byte aligned: 32 * 130 floats
    const SliceGroup g = sa.group[group];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cn = 8 * (g.pack1 - g.pack0);
    for (int i = tid; i < g.thr_n / 4; i += kSliceThreads)
        reinterpret_cast<float4 *>(st)[i] = __ldg(reinterpret_cast<const float4 *>(sa.thr + g.thr0) + i);
    int feat[kSliceRuns];
#pragma unroll
    for (int k = 0; k < kSliceRuns; ++k) {
        const int c = lane + 32 * k;
        feat[k] = c < cn ? __ldg(&sa.col[8 * g.pack0 + c].feature) : -1;
    }
    float next[kSliceRows][kSliceRuns];
    auto fetch = [&](int64_t b) {
#pragma unroll
        for (int r = 0; r < kSliceRows; ++r) {
            const int64_t row = 32 * b + warp + r * kSliceWarps;
            const float *src = X + row * ldx;
#pragma unroll
            for (int k = 0; k < kSliceRuns; ++k)
                next[r][k] = row < rows && feat[k] >= 0 ? __ldg(src + feat[k]) : 0.0f;
        }
    };
    if (b0 < b1) fetch(b0);
    for (int64_t b = b0; b < b1; b += step) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSliceRows; ++r)
#pragma unroll
            for (int k = 0; k < kSliceRuns; ++k)
                xs[(warp + r * kSliceWarps) * kSliceXs + lane + 32 * k] = next[r][k];
        __syncthreads();
        if (b + step < b1) fetch(b + step);
        const bool valid = 32 * b + lane < rows;
        for (int p = g.pack0 + warp; p < g.pack1; p += kSliceWarps) {
            const SlicePack pk = sa.pack[p];
            const int L = pk.levels;
            const float *tree = st + (pk.first - g.thr0);
            float x[8];
            int i[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                x[j] = xs[lane * kSliceXs + 8 * (p - g.pack0) + j];
                i[j] = 1;
            }
            for (int l = 0; l < L; ++l) {
#pragma unroll
                for (int j = 0; j < 8; ++j) i[j] = 2 * i[j] + (tree[(j << L) + i[j]] <= x[j] ? 1 : 0);
            }
            uint32_t w[3] = {0u, 0u, 0u};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                uint32_t c = (uint32_t)(i[j] - (1 << L));
                if (x[j] != x[j]) c = (uint32_t)__ldg(&sa.col[8 * p + j].count);
                if (!valid) c = 0u;
#pragma unroll
                for (int k = 0; k < 3; ++k) w[k] |= ((c >> (4 * k)) & 15u) << (4 * j);
            }
            uint32_t *dst = reinterpret_cast<uint32_t *>(codes) + ((size_t)b * sa.quads + 8 * p) * 4 + lane;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (4 * k < L) dst[(size_t)sa.qbase[k] * 4] = transpose32(w[k], lane);
        }
    }
}

__global__ void __launch_bounds__(kSliceThreads, 3) k_encode_slices(const float *__restrict__ X, int64_t rows,
                                                                   int64_t ldx, SliceArrays sa, int64_t blocks,
                                                                   unsigned char *__restrict__ codes) {
    extern __shared__ __align__(16) float slice_smem_raw[];
    early_launch();
    encode_group(X, rows, ldx, sa, blockIdx.y, blockIdx.x, blocks, gridDim.x, codes, slice_smem_raw);
}

// The rows of a ragged batch: item i = (request, group, first 32-row block, blocks); blocks
// walk the items.
__global__ void __launch_bounds__(kSliceThreads, 3) k_encode_batch(const ExplainJob *__restrict__ jobs,
                                                                  const BatchRequest *__restrict__ reqs,
                                                                  const int4 *__restrict__ items,
                                                                  const int *__restrict__ n_items) {
    extern __shared__ __align__(16) float slice_smem_raw[];
    const int count = n_items[0];
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const int4 it = items[i];
        const BatchRequest rq = reqs[it.x];
        const SliceArrays sa = jobs[rq.job].sa;
        encode_group(rq.C, rq.n, rq.ldc, sa, it.y, it.z, (int64_t)it.z + it.w, 1, rq.codes, slice_smem_raw);
        __syncthreads();
    }
}

int encode_batch_grid(int max_group_thr, const DevInfo &dev) {
    const size_t smem = slice_smem(max_group_thr);
    return dev.sms * (int)std::max<size_t>(1, std::min<size_t>(3, dev.smem_optin / (smem + 1024)));
}

cudaError_t launch_encode_batch(const ExplainJob *jobs, const BatchRequest *reqs, const int4 *items,
                                const int *n_items, int max_group_thr, const DevInfo &dev, cudaStream_t st) {
    const size_t smem = slice_smem(max_group_thr);
    cudaError_t err = allow_shared(k_encode_batch, smem, dev);
    if (err != cudaSuccess) return err;
    k_encode_batch<<<encode_batch_grid(max_group_thr, dev), kSliceThreads, smem, st>>>(jobs, reqs, items, n_items);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_encode_slices(const float *X, int64_t rows, int64_t ldx, const SliceArrays &sa, int64_t rows_pad,
                                 unsigned char *codes, const DevInfo &dev, cudaStream_t st) {
    const int64_t blocks = rows_pad / 32;
    if (blocks == 0) return cudaSuccess;
    const size_t smem = slice_smem(sa.max_group_thr);
    cudaError_t err = allow_shared(k_encode_slices, smem, dev);
    if (err != cudaSuccess) return err;
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(3, dev.smem_optin / (smem + 1024)));
    const int64_t fill = std::max<int64_t>(1, (int64_t)dev.sms * per_sm / sa.n_groups);
    dim3 grid((unsigned)std::min(blocks, fill), (unsigned)sa.n_groups);
    k_encode_slices<<<grid, kSliceThreads, smem, st>>>(X, rows, ldx, sa, blocks, codes);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace wdf
