// The step before the path: float weights -> per-channel scale alpha and ternary
// 2-bit codes (paper, Section 3.1, Eq. 1-3; Figure 10, pointwise branch).
//     alpha_i = mean_j |W[i][j]|,   W-hat[i][j] = clip(round(W[i][j] / max(alpha_i, eps)), -1, 1)
// with round = ties to even (the framework's), eps = 1e-5 guarding the division
// as in the figure.  Mean and ratio are taken in binary64, so that the order of
// the sum cannot move a decision at the precision of the float32 inputs.
// One warp per output channel (rows are a few hundred weights: a block per row spent its time in
// barriers and in the latency of two dependent reads, with too few rows in flight).  Latency is what
// bounds it, so a row of up to 1024 weights is read once and stays in registers, and a weight is coded
// by one comparison: clip(round(v), -1, 1) is 0 for |v| <= 1/2 (ties go to the even 0) and the sign
// otherwise, |W| * scale is monotone in |W|, so the row has one float threshold, found from the
// binary64 definition at the floats around mean / 2.  All 34 matrices of MobileNetV2 (9.1 MB, floor
// 1.4 us at the copy bandwidth), calls back to back: 10.3 us with two reads and binary64 decisions, 7.3 us now.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace prom { namespace quant {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;

// The largest |W| whose code is 0: |W| * scale, rounded to binary64, is at most 1/2 up to it and above
// for every larger float.  (mean / 2 is off by a few units in the last place at most.)
// A row with a weight that is not finite has no scale: its threshold, infinite or not a number, gives code 0 throughout.
__device__ __forceinline__ float zero_threshold(double mean, double scale)
{
    float t = (float)(0.5 * mean);
    for (int i = 0; i < 4 && (double)t * scale > 0.5; ++i) t = __int_as_float(__float_as_int(t) - 1);
    for (int i = 0; i < 4; ++i) {
        const float n = __int_as_float(__float_as_int(t) + 1);
        if (!((double)n * scale <= 0.5)) break;
        t = n;
    }
    return t;
}

// 2-bit code: 0, 1, or 3 for -1.  `bad` collects what is not finite (a NaN compares false).
__device__ __forceinline__ unsigned code_of(float w, float threshold, bool &bad)
{
    bad |= !(fabsf(w) <= 3.402823466e38f);
    return fabsf(w) > threshold ? 1u | (((unsigned)__float_as_int(w) >> 30) & 2u) : 0u;
}
__device__ __forceinline__ uint8_t code_byte(const float4 &v, float threshold, bool &bad)
{
    return (uint8_t)(code_of(v.x, threshold, bad) | (code_of(v.y, threshold, bad) << 2) |
                     (code_of(v.z, threshold, bad) << 4) | (code_of(v.w, threshold, bad) << 6));
}
__device__ __forceinline__ double abs_sum(const float4 &v)
{
    return (fabs((double)v.x) + fabs((double)v.y)) + (fabs((double)v.z) + fabs((double)v.w));
}

// One output channel (row) by one warp.  Every lane ends up with the same sum (butterfly), so the
// scale needs no exchange.
__device__ __forceinline__ void quantize_row(const float *__restrict__ row, int cin, double eps,
                                             uint8_t *__restrict__ packed_row, float *alpha_o)
{
    const int lane = threadIdx.x & 31;
    const int rowb = (cin + 3) >> 2;
    const bool vec = (cin & 3) == 0 && (reinterpret_cast<uintptr_t>(row) & 15u) == 0;
    const float4 *row4 = reinterpret_cast<const float4 *>(row);
    constexpr int kHeld = 8;                   // 8 x 32 lanes x 4 weights
    const bool held = vec && rowb <= kHeld * 32;
    float4 v[kHeld];
    double sum = 0.0;
    if (held) {
        // four weights = one 16-byte load = one byte of codes; all loads of the row are in flight at once
#pragma unroll
        for (int j = 0; j < kHeld; ++j) {
            v[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (lane + 32 * j < rowb) v[j] = __ldg(row4 + lane + 32 * j);
        }
#pragma unroll
        for (int j = 0; j < kHeld; ++j)
            if (32 * j < rowb) sum += abs_sum(v[j]);
    } else if (vec) {
#pragma unroll 4
        for (int kb = lane; kb < rowb; kb += 32) sum += abs_sum(__ldg(row4 + kb));
    } else {
        for (int j = lane; j < cin; j += 32) sum += fabs((double)row[j]);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
    const double mean = sum / (double)cin;
    if (alpha_o && lane == 0) *alpha_o = (float)mean;
    const double guarded = mean < eps ? eps : mean, scale = 1.0 / guarded;
    const float threshold = zero_threshold(guarded, scale);
    bool bad = false;
    if (held) {
#pragma unroll
        for (int j = 0; j < kHeld; ++j)
            if (lane + 32 * j < rowb) packed_row[lane + 32 * j] = code_byte(v[j], threshold, bad);
    } else if (vec) {
#pragma unroll 4
        for (int kb = lane; kb < rowb; kb += 32) packed_row[kb] = code_byte(__ldg(row4 + kb), threshold, bad);
    } else {
        for (int kb = lane; kb < rowb; kb += 32) {
            unsigned byte = 0;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = kb * 4 + e;
                if (k < cin) byte |= code_of(row[k], threshold, bad) << (2 * e);
            }
            packed_row[kb] = (uint8_t)byte;
        }
    }
    if (bad) raise_status(PROM_ERR_BAD_WEIGHT);
}

__global__ void __launch_bounds__(kThreads)
quantize_ternary_kernel(const float *__restrict__ w, int cout, int cin, double eps,
                        uint8_t *__restrict__ packed, float *__restrict__ alpha)
{
    ptx::grid_dep_wait();           // launched with programmatic dependent launch
    ptx::grid_dep_launch();
    const int rowb = (cin + 3) >> 2;
    const int warp = blockIdx.x * kWarps + (threadIdx.x >> 5), nwarps = gridDim.x * kWarps;
    for (int o = warp; o < cout; o += nwarps)
        quantize_row(w + (size_t)o * cin, cin, eps, packed + (size_t)o * rowb, alpha ? alpha + o : nullptr);
}

// Several weight matrices in one launch (all the layers of a network): the rows of all
// matrices are numbered through, and a block takes every gridDim.x-th of them.
constexpr int kMaxJobs = 64;
struct Jobs {
    int n;
    int first_row[kMaxJobs + 1];       // first global row of each matrix; first_row[n] = all rows
    int cin[kMaxJobs];
    const float *w[kMaxJobs];
    uint8_t *packed[kMaxJobs];
    float *alpha[kMaxJobs];
};

__global__ void __launch_bounds__(kThreads)
quantize_ternary_batch_kernel(const __grid_constant__ Jobs jobs, double eps)
{
    ptx::grid_dep_wait();           // launched with programmatic dependent launch
    ptx::grid_dep_launch();
    const int warp = blockIdx.x * kWarps + (threadIdx.x >> 5), nwarps = gridDim.x * kWarps;
    for (int r = warp; r < jobs.first_row[jobs.n]; r += nwarps) {
        int j = 0, end = jobs.n;               // the last matrix whose first row is at or before r
        while (end - j > 1) {
            const int mid = (j + end) >> 1;
            if (r >= jobs.first_row[mid]) j = mid; else end = mid;
        }
        const int o = r - jobs.first_row[j], cin = jobs.cin[j];
        quantize_row(jobs.w[j] + (size_t)o * cin, cin, eps, jobs.packed[j] + (size_t)o * ((cin + 3) >> 2),
                     jobs.alpha[j] ? jobs.alpha[j] + o : nullptr);
    }
}

}}  // namespace prom::quant
