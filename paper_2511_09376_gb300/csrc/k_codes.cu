// Decision codes (tree_layout.h) of a block of rows, in the 32-row code-block layout the
// decision kernels stage (wdf_device.cuh).
#include <algorithm>

#include "launch.h"
#include "wdf_device.cuh"

namespace wdf {

// Decision codes of rows [0, rows) of X into code blocks (wdf_device.cuh): element
// (block, column c, row r of block) at ((block * n_cols + c) * 32 + r) * code bytes.
// One thread block per 32-row code block: for every run of kEncodeCols columns the
// rows' values of the columns' features are read into shared memory (a warp reads
// along a row), then each warp encodes whole columns (lane = row).  Rows from rows to
// the end of the last block get code 0 (never counted).
constexpr int kEncodeThreads = 256;
constexpr int kEncodeCols = 128;  // 16.5 KB of staging: fits beside a counting block

// Code block `block` (rows 32 block .. 32 block + 31) of rows [0, rows) of X, written at
// codes + block * n_cols * 32 * code bytes.  xs: 32 x (kEncodeCols + 1) floats of shared
// memory.  All threads of the block call it.
__device__ __forceinline__ void encode_block(const float *__restrict__ X, int64_t rows, int64_t ldx,
                                             const TreeArrays &ta, int64_t block, unsigned char *__restrict__ codes,
                                             float *xs) {
    const int ncol = ta.n_cols, cb = ta.code_bytes;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row0 = block * 32;
    const bool valid = row0 + lane < rows;
    unsigned char *dst = codes + (size_t)block * ncol * 32 * cb;
    for (int c0 = 0; c0 < ncol; c0 += kEncodeCols) {
        const int cn = min(kEncodeCols, ncol - c0);
        __syncthreads();
        for (int r = warp; r < 32; r += kEncodeThreads / 32) {
            const int64_t row = row0 + r;
            for (int c = lane; c < cn; c += 32) {
                const int f = __ldg(&ta.cols[c0 + c].feature);
                xs[r * (kEncodeCols + 1) + c] = row < rows ? __ldg(X + row * ldx + f) : 0.0f;
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int c = warp; c < cn; c += kEncodeThreads / 32) {
            const int4 cv = __ldg(reinterpret_cast<const int4 *>(ta.cols) + c0 + c);
            const CodeCol col{cv.x, cv.y, cv.z, cv.w};
            const float x = xs[lane * (kEncodeCols + 1) + c];
            if (cb == 1) {
                // binary search from the column's top power of two (the same for the whole
                // warp) over its 255 padded entries: NaN padding is never <= x, so no bound
                // checks; a NaN x gets the count, as in decision_code
                const float *u = ta.col_thr + col.first;
                int pos = 0;
                for (int step = col.top; step > 0; step >>= 1) pos += __ldg(u + pos + step - 1) <= x ? step : 0;
                const int code = !valid ? 0 : (x != x ? col.count : pos);
                dst[(size_t)(c0 + c) * 32 + lane] = (unsigned char)code;
            } else {
                const int code = valid ? decision_code(x, ta.col_thr + col.first, col) : 0;
                reinterpret_cast<uint16_t *>(dst)[(size_t)(c0 + c) * 32 + lane] = (uint16_t)code;
            }
        }
    }
}

__global__ void __launch_bounds__(kEncodeThreads) k_encode_codes(const float *__restrict__ X, int64_t rows,
                                                                int64_t ldx, TreeArrays ta,
                                                                unsigned char *__restrict__ codes) {
    __shared__ float xs[32 * (kEncodeCols + 1)];
    encode_block(X, rows, ldx, ta, blockIdx.x, codes, xs);
}

// The rows of a ragged batch: item i = (request, 32-row block); blocks walk the items.
__global__ void __launch_bounds__(kEncodeThreads) k_encode_batch(const ExplainJob *__restrict__ jobs,
                                                                const BatchRequest *__restrict__ reqs,
                                                                const int2 *__restrict__ items,
                                                                const int *__restrict__ n_items) {
    __shared__ float xs[32 * (kEncodeCols + 1)];
    const int count = n_items[0];
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const int2 it = items[i];
        const BatchRequest rq = reqs[it.x];
        const TreeArrays ta = jobs[rq.job].ta;
        encode_block(rq.C, rq.n, rq.ldc, ta, it.y, rq.codes, xs);
    }
}

cudaError_t launch_encode_batch(const ExplainJob *jobs, const BatchRequest *reqs, const int2 *items,
                                const int *n_items, int grid, cudaStream_t st) {
    k_encode_batch<<<grid, kEncodeThreads, 0, st>>>(jobs, reqs, items, n_items);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_encode_codes(const float *X, int64_t rows, int64_t ldx, const TreeArrays &ta, int64_t rows_pad,
                                unsigned char *codes, cudaStream_t st) {
    const int64_t blocks = rows_pad / 32;
    if (blocks == 0) return cudaSuccess;
    k_encode_codes<<<(unsigned)blocks, kEncodeThreads, 0, st>>>(X, rows, ldx, ta, codes);
    count_launches(1);
    return cudaGetLastError();
}

// Sliced codes (tree_layout.h).  A block keeps the search trees of one group of packs in
// shared memory and walks 32-row blocks: the rows' values are read along the rows (the
// next block's while this one is searched), then a warp takes a pack of eight columns, lane
// = row: eight searches side by side (one shared load, compare and add per level; siblings
// of a level lie side by side, so lanes at different nodes of the first five levels read
// different banks), four bits of the eight codes packed into one word per lane, and a
// 32 x 32 bit transpose gives the pack's eight quads, written as 128 contiguous bytes.
// Issue-bound (76 %): 0.36 ms per 1M rows of 127 columns, where one byte per code and a
// search per (row, column) in global memory (k_encode_codes) takes 0.58 ms.
constexpr int kSliceThreads = 256, kSliceWarps = kSliceThreads / 32;
constexpr int kSliceCols = 8 * kSliceGroupPacks, kSliceXs = kSliceCols + 1;
constexpr int kSliceRows = 32 / kSliceWarps, kSliceRuns = kSliceCols / 32;

__global__ void __launch_bounds__(kSliceThreads, 3) k_encode_slices(const float *__restrict__ X, int64_t rows,
                                                                   int64_t ldx, SliceArrays sa, int64_t blocks,
                                                                   unsigned char *__restrict__ codes) {
    extern __shared__ __align__(16) float slice_smem[];
    float *xs = slice_smem, *st = slice_smem + 32 * kSliceXs + 32;  // 16-byte aligned: 32 * 130 floats
    const SliceGroup g = sa.group[blockIdx.y];
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
    if ((int64_t)blockIdx.x < blocks) fetch(blockIdx.x);
    for (int64_t b = blockIdx.x; b < blocks; b += gridDim.x) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSliceRows; ++r)
#pragma unroll
            for (int k = 0; k < kSliceRuns; ++k)
                xs[(warp + r * kSliceWarps) * kSliceXs + lane + 32 * k] = next[r][k];
        __syncthreads();
        if (b + gridDim.x < blocks) fetch(b + gridDim.x);
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

cudaError_t launch_encode_slices(const float *X, int64_t rows, int64_t ldx, const SliceArrays &sa, int64_t rows_pad,
                                 unsigned char *codes, const DevInfo &dev, cudaStream_t st) {
    const int64_t blocks = rows_pad / 32;
    if (blocks == 0) return cudaSuccess;
    const size_t smem = ((size_t)32 * kSliceXs + 32 + (size_t)sa.max_group_thr) * 4;
    if (smem > dev.smem_optin) return cudaErrorInvalidConfiguration;
    cudaError_t err = cudaFuncSetAttribute(k_encode_slices, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(3, dev.smem_optin / (smem + 1024)));
    const int64_t fill = std::max<int64_t>(1, (int64_t)dev.sms * per_sm / sa.n_groups);
    dim3 grid((unsigned)std::min(blocks, fill), (unsigned)sa.n_groups);
    k_encode_slices<<<grid, kSliceThreads, smem, st>>>(X, rows, ldx, sa, blocks, codes);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace wdf
