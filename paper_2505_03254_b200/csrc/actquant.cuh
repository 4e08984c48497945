// The step after the path in the paper's dataflow: per-sample absmax quantisation of float
// activations to int8 (paper, Section 3.1 "Activations", Eq. 6-7, and the activation figure of
// the pseudocode appendix):
//     gamma_i = max |X[i][...]|,  scale_i = 127 / max(gamma_i, eps),
//     X-hat[i][...] = clip(round(X[i][...] * scale_i), -128, 127)
// with round = ties to even and eps = 1e-5 guarding the division as in the figure.  The
// quotient and the product are single correctly rounded binary32 operations (__fdiv_rn,
// __fmul_rn: no contraction, no approximate division), the precision the paper's framework
// computes in, so the codes do not depend on how the work is split.
//
// Three routes.  Fused: a thread-block cluster per sample; every CTA copies its slice of the
// sample into shared memory once (bulk copies), the CTAs exchange their maxima through
// distributed shared memory, and the slice is quantised from shared memory: each float is read
// from HBM once (5 bytes per element).  Grouped: the codes of one group of samples, which L2 still
// holds, and then the maxima of the next (samples that do not fit eight SMs' shared memory, and batches
// of which clusters would take several rounds).  Two-pass, for sizes that are not a multiple of 4: one kernel
// takes the maxima with atomicMax on the bit pattern, a second one quantises.
// Measured, calls back to back (floor: 5 bytes per value at the copy bandwidth): [128,112,112,32] 58 us (39; 64
// before chunks were held in registers, 74.5 when a lane quantised 64 neighbouring bytes and met four-way bank conflicts); [1,112,112,320] 8 us
// (3; 60 on one cluster); [60,112,112,96] 96 us (55; 107); [192,7,7,960] 11 us (7; 19).
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"
#include "ptx.cuh"

namespace prom { namespace actq {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;
constexpr int kMaxCluster = 8;
constexpr unsigned long long kWaitLimitNs = 100000000ull;
constexpr uint32_t kCopyBytes = 32768;          // one bulk copy
constexpr int kMaxChunks = 8;                   // 8 x 32 KB >= the shared memory of an SM

// round(x * sc) as an integer, ties to even: adding 1.5 * 2^23 rounds the sum to a whole number
// in one correctly rounded binary32 addition, and the whole number sits in the low mantissa
// bits.  Exact for |x * sc| < 2^22; |x| <= gamma keeps the product at 127 (plus rounding).
__device__ __forceinline__ int round_scaled(float x, float sc)
{
    const float r = __fadd_rn(__fmul_rn(x, sc), 12582912.0f);
    return __float_as_int(r) - 0x4B400000;
}

__device__ __forceinline__ int8_t quantise_one(float x, float sc)
{
    int r = round_scaled(x, sc);
    r = r > 127 ? 127 : (r < -128 ? -128 : r);
    return (int8_t)r;
}

// four codes in one word: saturating packs clip to [-128, 127]
__device__ __forceinline__ uint32_t quantise_four(const float4 v, float sc)
{
    uint32_t w;
    asm("{\n\t.reg .b32 t;\n\t"
        "cvt.pack.sat.s8.s32.b32 t, %4, %3, 0;\n\t"
        "cvt.pack.sat.s8.s32.b32 %0, %2, %1, t;\n\t}"
        : "=r"(w)
        : "r"(round_scaled(v.x, sc)), "r"(round_scaled(v.y, sc)), "r"(round_scaled(v.z, sc)),
          "r"(round_scaled(v.w, sc)));
    return w;
}

__device__ __forceinline__ float scale_of(float gamma, float eps)
{
    return __fdiv_rn(127.0f, gamma < eps ? eps : gamma);
}

// max |x| over a block; every thread gets the result.  NaNs are skipped (a > m is false).
__device__ __forceinline__ float block_absmax(float m, float *part)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const float o = __shfl_xor_sync(0xFFFFFFFFu, m, d);
        m = o > m ? o : m;
    }
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    float r = 0.0f;
    for (int i = 0; i < kThreads / 32; ++i) r = part[i] > r ? part[i] : r;
    __syncthreads();
    return r;
}

// Fused route.  The grid is as many clusters as the GPU holds at once; cluster k takes samples
// k, k + clusters, ...  CTA r of a cluster owns floats [r * slice, min(per, (r + 1) * slice)) of
// each of them; slice is a multiple of 16 and slice * 4 bytes fit the dynamic shared memory.
// The slice arrives in chunks of kCopyBytes, one mbarrier each: the maximum of a chunk is taken
// while later chunks are on their way, and as soon as a chunk has been quantised its place is
// filled with the same chunk of the cluster's next sample.
// HOLD: the first chunks of a sample stay in registers once their maximum is taken, 16 floats per thread and chunk,
// and their places are filled at once.  Without that no copy is on its way from the last chunk's arrival over the
// exchange to the first code, about 2 of the 8 us that a round of samples took.  It costs 48 registers for the three
// chunks (96 KB) that cover the gap, so it is for slices that fill an SM; smaller ones share it.  (128 samples of 1.6 MB:
// 64.0 us without, 61.4, 59.3, 58.0, 58.4 and 60.6 with one to five chunks.)
template <int HOLD>
__global__ void __launch_bounds__(kThreads, 1)
act_quant_cluster_kernel(const float *__restrict__ x, int batch, long long per, int slice, float eps,
                         int8_t *__restrict__ q, float *__restrict__ gamma, float *__restrict__ scale)
{
    extern __shared__ __align__(128) uint8_t smem_raw[];
    float *buf = reinterpret_cast<float *>(smem_raw);
    __shared__ float part[kThreads / 32];
    __shared__ float peer_max[2][kMaxCluster];
    __shared__ __align__(8) uint64_t bar[kMaxChunks];
    __shared__ int failed;

    cg::cluster_group cluster = cg::this_cluster();
    const unsigned rank = cluster.block_rank(), csize = cluster.num_blocks();
    const int cid = blockIdx.x / csize, nclusters = gridDim.x / csize;
    const long long first = (long long)rank * slice;
    long long count = per - first;
    count = count < 0 ? 0 : (count > slice ? slice : count);        // floats of this CTA
    const uint32_t bytes = (uint32_t)count * 4u;
    const int nchunks = (int)((bytes + kCopyBytes - 1) / kCopyBytes);
    const uint32_t bar_addr = ptx::smem_u32(&bar[0]);
    const uint32_t buf_addr = ptx::smem_u32(buf);
    const float4 *b4 = reinterpret_cast<const float4 *>(buf);
    // every CTA of the cluster must be running before another one writes into its shared
    // memory: arrive now, wait just before the first exchange
    cluster.barrier_arrive();
    // launched with programmatic dependent launch: x may be the previous kernel's output
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    auto load_chunk = [&](int sample, int c) {      // thread 0 only
        const uint8_t *src = reinterpret_cast<const uint8_t *>(x + (long long)sample * per + first);
        const uint32_t off = (uint32_t)c * kCopyBytes;
        const uint32_t len = bytes - off < kCopyBytes ? bytes - off : kCopyBytes;
        ptx::mbar_expect_tx(bar_addr + 8 * c, len);
        ptx::bulk_load(buf_addr + off, src + off, len, bar_addr + 8 * c);
    };
    if (threadIdx.x == 0) {
        failed = 0;
        for (int c = 0; c < nchunks; ++c) ptx::mbar_init(bar_addr + 8 * c, 1);
        ptx::mbar_init_fence();
        if (cid < batch)
            for (int c = 0; c < nchunks; ++c) load_chunk(cid, c);
    }
    __syncthreads();

    bool ok = true;
    bool first_exchange = true;
    uint32_t parity = 0;
    constexpr int kPer = (int)(kCopyBytes / 16) / kThreads;       // 16-byte words of a chunk per thread
    float4 held[HOLD > 0 ? HOLD * kPer : 1];
    for (int sample = cid, it = 0; sample < batch; sample += nclusters, ++it, parity ^= 1u) {
        const int next = sample + nclusters;
        // ---- this CTA's maximum, chunk by chunk as the copies land (bounded waits) --------
        float m = 0.0f;
        auto landed = [&](int c) {
            unsigned long long t0 = 0;
            for (uint32_t i = 1; !ptx::mbar_try_wait(bar_addr + 8 * c, parity); ++i) {
                if ((i & 255u) == 0) {
                    const unsigned long long now = ptx::globaltimer();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > kWaitLimitNs) return false;
                }
            }
            return true;
        };
#pragma unroll
        for (int c = 0; c < HOLD; ++c) {
            if (c >= nchunks) break;
            ok = ok && landed(c);
            const int lo = c * (int)(kCopyBytes / 16), hi = min((int)(count >> 2), lo + (int)(kCopyBytes / 16));
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int i = lo + (int)threadIdx.x + j * kThreads;
                const float4 v = ok && i < hi ? b4[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                held[kPer * c + j] = v;
                float a = fabsf(v.x); m = a > m ? a : m;
                a = fabsf(v.y); m = a > m ? a : m;
                a = fabsf(v.z); m = a > m ? a : m;
                a = fabsf(v.w); m = a > m ? a : m;
            }
            __syncthreads();              // the chunk has been read by everyone
            if (threadIdx.x == 0 && ok && next < batch) load_chunk(next, c);
        }
        for (int c = HOLD; c < nchunks && ok; ++c) {
            ok = landed(c);
            if (!ok) break;
            const int lo = c * (int)(kCopyBytes / 16);
            const int hi = min((int)(count >> 2), lo + (int)(kCopyBytes / 16));
            for (int i = lo + threadIdx.x; i < hi; i += kThreads) {
                const float4 v = b4[i];
                float a = fabsf(v.x); m = a > m ? a : m;
                a = fabsf(v.y); m = a > m ? a : m;
                a = fabsf(v.z); m = a > m ? a : m;
                a = fabsf(v.w); m = a > m ? a : m;
            }
        }
        if (!ok && !failed) {
            failed = 1;                   // any thread that gave up marks the CTA; the cluster
            raise_status(PROM_ERR_TIMEOUT);   // barriers below are still taken, so nobody hangs
        }
        m = block_absmax(m, part);        // two block-wide syncs inside
        ok = failed == 0;

        // ---- every CTA's maximum to every CTA ---------------------------------------------
        if (first_exchange) { cluster.barrier_wait(); first_exchange = false; }
        if (threadIdx.x < csize) *cluster.map_shared_rank(&peer_max[it & 1][rank], threadIdx.x) = m;
        cluster.sync();
        float g = 0.0f;
        for (unsigned r = 0; r < csize; ++r) g = peer_max[it & 1][r] > g ? peer_max[it & 1][r] : g;
        const float sc = scale_of(g, eps);
        if (rank == 0 && threadIdx.x == 0) {
            gamma[sample] = g;
            scale[sample] = sc;
        }

        // ---- quantise from shared memory; refill each chunk at once ----
        int8_t *dst = q + (long long)sample * per + first;
#pragma unroll
        for (int c = 0; c < HOLD; ++c) {
            if (!ok || c >= nchunks) break;
            const int lo = c * (int)(kCopyBytes / 16), hi = min((int)(count >> 2), lo + (int)(kCopyBytes / 16));
            uint32_t *dst4 = reinterpret_cast<uint32_t *>(dst);
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int i = lo + (int)threadIdx.x + j * kThreads;
                if (i < hi) dst4[i] = quantise_four(held[kPer * c + j], sc);
            }
        }
        for (int c = HOLD; c < nchunks; ++c) {
            if (ok) {
                // (four codes per thread: neighbouring lanes on neighbouring 16-byte words, no bank conflicts)
                const int lo = c * (int)(kCopyBytes / 16);
                const int hi = min((int)(count >> 2), lo + (int)(kCopyBytes / 16));
                uint32_t *dst4 = reinterpret_cast<uint32_t *>(dst);
#pragma unroll 4
                for (int i = lo + threadIdx.x; i < hi; i += kThreads) dst4[i] = quantise_four(b4[i], sc);
            }
            __syncthreads();              // the chunk has been read by everyone
            if (threadIdx.x == 0 && ok && next < batch) load_chunk(next, c);
        }
    }
    if (first_exchange) cluster.barrier_wait();     // a cluster without a sample still pairs its arrive
    if (HOLD > 0 && threadIdx.x == 0 && failed) {   // copies may be on their way for a sample that is not awaited any more
        const unsigned long long t0 = ptx::globaltimer();
        while (ptx::globaltimer() - t0 < kWaitLimitNs) {}
    }
}

// Grouped route.  The samples are taken in groups of up to 64 MB, kernel k of the call quantises group k - 1, whose
// maxima kernel k - 1 took and which L2 still holds, and then takes the maxima of group k: HBM reads a float once, and
// every SM works on every group whatever the number and size of the samples.  (The other way round, so that maxima ran
// beside the codes of the kernel in front, L2 had to hold two groups: 33 samples of 34.5 MB took 469 us in groups of one
// sample, now 404; 33 of 11.7 MB 139 in groups of 40 MB, now 116.)  A warp takes a contiguous run of pieces of kPiece
// floats, a piece lies in one sample; per is a multiple of 4.
constexpr int kGroupThreads = 512;
constexpr int kPieceVec = 8;                        // float4 loads of a lane in flight
constexpr int kPiece = 32 * 4 * kPieceVec;
struct GroupArgs {
    const float *x;
    long long per;
    long long pieces;           // of a sample
    int max_first, max_count;   // samples whose maxima are taken
    int q_first, q_count;       // samples that are quantised
    int first;                  // the first kernel of the call
    float eps;
    int8_t *q;
    float *gamma, *scale;
};

// This warp's run [p, end) of `total` pieces.
__device__ __forceinline__ void warp_run(long long total, long long &p, long long &end)
{
    const long long warps = (long long)gridDim.x * (kGroupThreads / 32);
    const long long w = (long long)blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5);
    const long long each = total / warps, more = total % warps;
    p = w * each + (w < more ? w : more);
    end = p + each + (w < more ? 1 : 0);
}

__device__ __forceinline__ void group_maxima(const GroupArgs &a)
{
    const int lane = threadIdx.x & 31;
    const long long per4 = a.per >> 2;
    long long p, end;
    warp_run(a.pieces * a.max_count, p, end);
    if (p >= end) return;
    long long s = p / a.pieces, r = p - s * a.pieces;
    float m = 0.0f;
    for (; p < end; ++p) {
        const float4 *src = reinterpret_cast<const float4 *>(a.x + (a.max_first + s) * a.per) + r * (kPiece / 4);
        const int left = (int)(per4 - r * (kPiece / 4) < kPiece / 4 ? per4 - r * (kPiece / 4) : kPiece / 4);
        float4 v[kPieceVec];
#pragma unroll
        for (int j = 0; j < kPieceVec; ++j)
            v[j] = lane + 32 * j < left ? __ldg(src + lane + 32 * j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int j = 0; j < kPieceVec; ++j)       // (fmaxf drops NaNs)
            m = fmaxf(fmaxf(m, fmaxf(fabsf(v[j].x), fabsf(v[j].y))), fmaxf(fabsf(v[j].z), fabsf(v[j].w)));
        if (++r == a.pieces || p + 1 == end) {
            // non-negative floats are ordered like their bit patterns
            const uint32_t g = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(m));
            if (lane == 0 && g) atomicMax(reinterpret_cast<unsigned int *>(a.gamma + a.max_first + s), g);
            m = 0.0f;
            if (r == a.pieces) { r = 0; ++s; }
        }
    }
}

__device__ __forceinline__ void group_codes(const GroupArgs &a)
{
    const int lane = threadIdx.x & 31;
    const long long per4 = a.per >> 2;
    long long p, end;
    warp_run(a.pieces * a.q_count, p, end);
    if (p >= end) return;
    long long s = p / a.pieces, r = p - s * a.pieces;
    float sc = 0.0f;
    bool fresh = true;
    for (; p < end; ++p) {
        const long long sample = a.q_first + s, at = r * (kPiece / 4);
        const float4 *src = reinterpret_cast<const float4 *>(a.x + sample * a.per) + at;
        uint32_t *dst = reinterpret_cast<uint32_t *>(a.q + sample * a.per) + at;
        const int left = (int)(per4 - at < kPiece / 4 ? per4 - at : kPiece / 4);
        float4 v[kPieceVec];
#pragma unroll
        for (int j = 0; j < kPieceVec; ++j)
            if (lane + 32 * j < left) v[j] = __ldcs(src + lane + 32 * j);
        if (fresh) {
            sc = scale_of(__ldcg(a.gamma + sample), a.eps);
            if (r == 0 && lane == 0) a.scale[sample] = sc;
            fresh = false;
        }
#pragma unroll
        for (int j = 0; j < kPieceVec; ++j)
            if (lane + 32 * j < left) __stcs(dst + lane + 32 * j, quantise_four(v[j], sc));
        if (++r == a.pieces) { r = 0; ++s; fresh = true; }
    }
}

// SEVERAL: the call has more than one group.  (With one, a kernel does either the one or the other, and the shorter way
// to the maxima is worth 2 to 4 % of 12 us.)
template <bool SEVERAL>
__global__ void __launch_bounds__(kGroupThreads, 2) act_group_kernel(const GroupArgs a)
{
    // The first kernel waits for what wrote x and for the cleared maxima, the others for the maxima of the group before.
    if (a.first) ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (SEVERAL) {
        if (!a.first) ptx::grid_dep_wait();
        group_codes(a);
        group_maxima(a);
    } else {
        group_maxima(a);
        if (!a.first) ptx::grid_dep_wait();
        group_codes(a);
    }
}

// Two-pass route, pass 1: gamma (zeroed beforehand) takes the maxima; |x| >= 0, so the order of
// the bit patterns is the order of the values.
__global__ void __launch_bounds__(kThreads)
act_absmax_kernel(const float *__restrict__ x, long long per, float *__restrict__ gamma)
{
    __shared__ float part[kThreads / 32];
    const long long sample = blockIdx.y;
    const float *src = x + sample * per;
    float m = 0.0f;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < per; i += (long long)gridDim.x * kThreads) {
        const float a = fabsf(src[i]);
        m = a > m ? a : m;
    }
    m = block_absmax(m, part);
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned int *>(gamma + sample), __float_as_uint(m));
}

// Two-pass route, pass 2.
__global__ void __launch_bounds__(kThreads)
act_quant_kernel(const float *__restrict__ x, long long per, float eps, const float *__restrict__ gamma,
                 int8_t *__restrict__ q, float *__restrict__ scale)
{
    const long long sample = blockIdx.y;
    const float sc = scale_of(gamma[sample], eps);
    if (blockIdx.x == 0 && threadIdx.x == 0) scale[sample] = sc;
    const float *src = x + sample * per;
    int8_t *dst = q + sample * per;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < per; i += (long long)gridDim.x * kThreads)
        dst[i] = quantise_one(src[i], sc);
}

}}  // namespace prom::actq
