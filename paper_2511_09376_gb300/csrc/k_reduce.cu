// Global attribution: per-feature means of |phi| and phi over many explained rows,
// accumulated in FP64 (the paper's global attribution combines many local
// attributions, section "Introduction").  Two passes with a fixed summation order, so
// the result does not depend on scheduling: row blocks write FP64 partial sums, then
// 32 threads per feature add them.
#include <algorithm>
#include <cstdint>

#include "launch.h"

namespace wdf {

constexpr int kRowsPerBlock = 4096;  // of the general form

// The packed form: as many blocks as two per SM of 152, fewer for few rows, and never more
// partial sums than kPackedPartials (what the allocation-free entry point holds).
constexpr int kVecMaxF = 512, kVecBlocks = 304, kVecMinRows = 32;
constexpr int64_t kPackedPartials = (int64_t)1 << 18;

static int64_t packed_rows(int64_t n, int F) {  // rows per block, a multiple of 4
    const int64_t most = std::min<int64_t>(kVecBlocks, kPackedPartials / (2 * F));
    return std::max<int64_t>(kVecMinRows, ((n + most - 1) / most + 3) & ~(int64_t)3);
}

static int64_t packed_blocks(int64_t n, int F) { return std::max<int64_t>(1, (n + packed_rows(n, F) - 1) / packed_rows(n, F)); }

int64_t global_attr_blocks(int64_t n) { return std::max<int64_t>(1, (n + kRowsPerBlock - 1) / kRowsPerBlock); }

int64_t global_attr_partial_doubles(int64_t n, int F) {
    return std::max(global_attr_blocks(n), F <= kVecMaxF ? packed_blocks(n, F) : (int64_t)0) * (int64_t)F * 2;
}

// block (32, 8): column f = 32 * blockIdx.y + threadIdx.x, row sub-lane threadIdx.y.
// The general form (any row stride and alignment).
__global__ void __launch_bounds__(256) k_colsum_partial(const float *__restrict__ phi, int64_t n, int64_t ldp, int F,
                                                        double *__restrict__ partial) {
    __shared__ double sa[8][32], ss[8][32];
    const int f = blockIdx.y * 32 + threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * kRowsPerBlock;
    const int64_t r1 = (n < r0 + kRowsPerBlock) ? n : r0 + kRowsPerBlock;
    double a = 0.0, s = 0.0;
    if (f < F) {
        for (int64_t r = r0 + threadIdx.y; r < r1; r += 8) {
            const double v = (double)__ldg(phi + r * ldp + f);
            a += fabs(v);
            s += v;
        }
    }
    sa[threadIdx.y][threadIdx.x] = a;
    ss[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && f < F) {
        double ta = 0.0, ts = 0.0;
        for (int k = 0; k < 8; ++k) {
            ta += sa[k][threadIdx.x];
            ts += ss[k][threadIdx.x];
        }
        partial[((size_t)blockIdx.x * F + f) * 2 + 0] = ta;
        partial[((size_t)blockIdx.x * F + f) * 2 + 1] = ts;
    }
}

// Packed rows (row stride F, 16-byte aligned) with F <= kVecMaxF: the block's rows are one
// flat run of floats read as float4.  Threads = F * c, so 4 * threads is a multiple of F and
// thread t always meets features (4t + j) mod F, j = 0..3.
//
// FP64 adds and conversions run at two a clock and SM on this GPU, so the sums stay in FP32
// without giving up FP64 results:
//  - A run of kRun elements of a column is cut twice at common powers of two.  With 2^e the
//    largest magnitude's binade and M = 1.5 * 2^(e + 4), q = (x + M) - M is x rounded to a
//    multiple of 2^(e - 19), so the run's sum of q (and of |q|) is exact.  The rest r = x - q is
//    exact too and at most 2^(e - 20); cut the same way at multiples of 2^(e - 40) its sum is
//    exact as well.  What is then left of an element is exact, at most 2^(e - 41), and zero for all
//    elements of 2^(e - 17) and more; its plain sum is within 2^(e - 57) of the run's (15
//    additions of partial sums of at most 2^(e - 37), each off by at most 2^-24 of its result).
//    q and the rests carry x's sign into the sum of magnitudes.
//  - The run's three parts go into a thread's sum of three FP32 (h + m + l by error-free
//    TwoSum, the last plain), some 2^-60 of it, and that into FP64 once per thread.
// So a thread's sum is FP64's but for its last rounding.  (With one cut and a plain sum of r, one
// large element and fifteen just below 2^-20 of it were 6e-14 of the mean off.)
// Elements of 2^123 and more, infinities and NaN take plain FP64 sums over the thread's
// elements instead (nothing above is exact for them).
// Bound by reading phi: 1,000,000 x 127 (508 MB), the whole call: 94 us (5.4 TB/s), 88 with one cut,
// 380 with two FP64 adds per eight elements and sum and 1.6 waves of blocks.  Two blocks of 254
// threads per SM keep 130 KB of loads in flight, so one wave of 304 blocks is enough.
constexpr int kRun = 16;
constexpr uint32_t kRunShift = 4;    // log2 kRun
constexpr uint32_t kRestShift = 17;  // the second cut's M: 1.5 * 2^(e - 17) (below 2^-109 of FP32's range every r is cut to itself)

struct Sum3 {
    float h = 0.0f, m = 0.0f, l = 0.0f;
    __device__ __forceinline__ static float two_sum(float &s, float x) {  // s += x; returns the error
        const float t = s + x, b = t - s;
        const float e = (s - (t - b)) + (x - b);
        s = t;
        return e;
    }
    __device__ __forceinline__ void add(float q, float r, float rest) {
        l += two_sum(m, two_sum(h, q));
        l += two_sum(m, r);
        l += rest;
    }
    __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
};

__global__ void __launch_bounds__(kVecMaxF, 1) k_colsum_vec(const float *__restrict__ phi, int64_t n, int F,
                                                             int64_t rows, double *__restrict__ partial) {
    __shared__ double sa[4 * kVecMaxF], ss[4 * kVecMaxF];
    const int NT = blockDim.x, t = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * rows;
    const int64_t r1 = (n < r0 + rows) ? n : r0 + rows;
    const float *base = phi + r0 * F;  // 16-byte aligned: r0 is a multiple of 4
    const int64_t nel = (r1 - r0) * F, nq = nel / 4;
    const float4 *b4 = reinterpret_cast<const float4 *>(base);
    Sum3 A[4], S[4];
    float top = 0.0f;
    for (int64_t q0 = t; q0 < nq; q0 += (int64_t)kRun * NT) {
        float4 v[kRun];
        const float4 *src = b4 + q0;
        if (q0 + (int64_t)(kRun - 1) * NT < nq) {
#pragma unroll
            for (int k = 0; k < kRun; ++k) v[k] = __ldcs(src + k * NT);
        } else {
#pragma unroll
            for (int k = 0; k < kRun; ++k)
                v[k] = q0 + (int64_t)k * NT < nq ? __ldcs(src + k * NT) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float x[kRun], mx = 0.0f;
#pragma unroll
            for (int k = 0; k < kRun; ++k) {
                x[k] = j == 0 ? v[k].x : j == 1 ? v[k].y : j == 2 ? v[k].z : v[k].w;
                mx = fmaxf(mx, fabsf(x[k]));
            }
            top = fmaxf(top, mx);
            const uint32_t e = __float_as_uint(mx) & 0x7F800000u, e2 = max(e, kRestShift << 23) - (kRestShift << 23);
            const float M = __uint_as_float(e + (kRunShift << 23) + 0x00400000u), M2 = __uint_as_float(e2 + 0x00400000u);
            float q1 = 0.0f, qa = 0.0f, r1 = 0.0f, ra = 0.0f, d1 = 0.0f, da = 0.0f;
#pragma unroll
            for (int k = 0; k < kRun; ++k) {
                const float sign = __uint_as_float((__float_as_uint(x[k]) & 0x80000000u) | 0x3F800000u);
                const float q = (x[k] + M) - M, rest = x[k] - q, r = (rest + M2) - M2, d = rest - r;
                q1 += q;
                qa += fabsf(q);
                r1 += r;
                ra = fmaf(r, sign, ra);
                d1 += d;
                da = fmaf(d, sign, da);
            }
            S[j].add(q1, r1, d1);
            A[j].add(qa, ra, da);
        }
    }
    double sum[4], mag[4];
    bool plain = !(top < 0x1p123f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        sum[j] = S[j].value();
        mag[j] = A[j].value();
        plain |= !(fabs(mag[j]) <= 1.7976931348623157e308);  // NaN, or a sum beyond FP32
    }
    if (plain) {
#pragma unroll
        for (int j = 0; j < 4; ++j) sum[j] = mag[j] = 0.0;
        for (int64_t q = t; q < nq; q += NT) {
            const float4 v = __ldg(b4 + q);
            const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mag[j] += fabs((double)x[j]);
                sum[j] += (double)x[j];
            }
        }
    }
    // the last (nel mod 4) elements belong to the slots of the thread that owns float4 nq
    if (t == (int)(nq % NT)) {
        const int tail = (int)(nel - 4 * nq);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (j < tail) {
                const double x = (double)__ldg(base + 4 * nq + j);
                mag[j] += fabs(x);
                sum[j] += x;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        sa[4 * t + j] = mag[j];
        ss[4 * t + j] = sum[j];
    }
    __syncthreads();
    const int c4 = 4 * NT / F;
    for (int f = t; f < F; f += NT) {
        double ta = 0.0, ts = 0.0;
        for (int i = 0; i < c4; ++i) {
            ta += sa[f + F * i];
            ts += ss[f + F * i];
        }
        reinterpret_cast<double2 *>(partial)[(size_t)blockIdx.x * F + f] = make_double2(ta, ts);
    }
}

// The blocks' partial sums, in a fixed order: eight features per block, 32 threads each
// (7 us for 304 x 127; a thread per feature took 30 us for 245 x 127, one load after another).
__global__ void __launch_bounds__(256) k_colsum_final(const double *__restrict__ partial, int nb, int F, int64_t n,
                                                      double *__restrict__ mean_abs, double *__restrict__ mean) {
    __shared__ double sa[32][8], ss[32][8];
    const int c = threadIdx.x & 7, y = threadIdx.x >> 3, f = blockIdx.x * 8 + c;
    double ta = 0.0, ts = 0.0;
    if (f < F) {
#pragma unroll 4
        for (int b = y; b < nb; b += 32) {
            const double2 p = __ldg(reinterpret_cast<const double2 *>(partial) + (size_t)b * F + f);
            ta += p.x;
            ts += p.y;
        }
    }
    sa[y][c] = ta;
    ss[y][c] = ts;
    for (int k = 16; k > 0; k >>= 1) {
        __syncthreads();
        if (y < k) {
            sa[y][c] += sa[y + k][c];
            ss[y][c] += ss[y + k][c];
        }
    }
    if (y > 0 || f >= F) return;
    const double inv = n > 0 ? 1.0 / (double)n : 0.0;
    mean_abs[f] = sa[0][c] * inv;
    mean[f] = ss[0][c] * inv;
}

cudaError_t launch_global_attr(const float *phi, int64_t n, int64_t ldp, int F, double *partial, double *mean_abs,
                               double *mean, cudaStream_t st) {
    const bool vec = ldp == F && F <= kVecMaxF && (reinterpret_cast<uintptr_t>(phi) & 15) == 0;
    const int64_t nb64 = vec ? packed_blocks(n, F) : global_attr_blocks(n);
    if (nb64 > 0x7FFFFFFF) return cudaErrorInvalidValue;
    const int nb = (int)nb64;
    if (n > 0) {
        if (vec) {
            const int threads = F * std::max(1, 256 / F);
            k_colsum_vec<<<nb, threads, 0, st>>>(phi, n, F, packed_rows(n, F), partial);
        } else {
            dim3 grid(nb, (F + 31) / 32);
            k_colsum_partial<<<grid, dim3(32, 8), 0, st>>>(phi, n, ldp, F, partial);
        }
        count_launches(1);
        cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return err;
    }
    k_colsum_final<<<(F + 7) / 8, 256, 0, st>>>(partial, n > 0 ? nb : 0, F, n, mean_abs, mean);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace wdf
