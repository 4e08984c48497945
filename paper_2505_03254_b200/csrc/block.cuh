// A whole inverted-residual block in one launch: the expanding pointwise layer, the depthwise 3x3
// convolution (stride 1 or 2) and the projecting pointwise layer with its skip connection.  The expanded
// tensor, six times as wide as the block's input, and the depthwise output exist a slice of 64 channels
// at a time in shared memory and are never written.
//
// Work decomposition
//   item   = a band of `rows` output rows of one image (or `ipi` whole images of a small plane)
//   slice  = 64 expanded channels
//   unit   = 128 pixels of a slice: one accumulator of 128 lanes x 64 columns
// A CTA takes an item through its slices; for every slice
//   E   its input pixels (with the halo rows) times the slice's expand weights, requantised into a pixel
//       buffer: pixel (row r, column x) at index r * pitch + x + 1, 64 bytes each, pitch = width + 1, the
//       pixel between two rows being the zero padding of both.  In that order a tap of the depthwise
//       convolution is nothing but an offset: output i = row * pitch + column reads i + dy * pitch + dx.
//       (Stride 2: four such planes, of even and odd rows and columns.)
//   D   nine MMAs of 128 x 32 x 32 per 128 outputs of 32 channels, A the pixel buffer at the tap's offset, B the
//       tap's weights on a diagonal, and one for the bias; requantised into a 128 x 64 operand block
//   P   that block times the slice's project weights, accumulated over the slices in tensor memory.
// With few items the slices are split over the CTAs of a cluster, whose 32-bit sums are exchanged through
// distributed shared memory, each CTA requantising a share of the pixels.
//
// Roles: warp 0 loads the slices' prepared operands (one bulk copy each) and input pixels, warps 1, 2 and 3
// issue the MMAs of E, D and P, warps 4.. are four groups of four epilogue warps that take units in the
// order E(k + ahead, all), D(k, all), so that the expansion of slices overlaps the depthwise part of those
// before.  Every wait is for something earlier in that order, which is the same in all roles.
// Units of a kind go to the groups in turn.  Barriers of units and slices are rings of eight, whatever the
// number of buffers behind them: a group that waits for a unit has waited for the one `groups` before it, so
// the barrier it looks at cannot be a whole turn behind.
//
// What bounds it: with many units a slice of D, 20 MMAs that read 5 KB of shared memory each, 800 cycles alone and
// about 1500 beside the epilogue's constants and stores; with few, the chain load, E, D, P, exchange (about 8 us) and
// what lies between two launches (2.5 to 3.5 us, since a CTA fills the SM).  Measured inside the network's body, us, one
// launch per layer -> one per block: batch 9 at width 0.75: 56 x 56 x 24 -> 144 -> 24 19.4 -> 13.3, 28 x 28 x 24 -> 144 -> 24
// 12.3 -> 9.0, 14 x 14 x 72 -> 432 -> 72 12.9 -> 11.0, 7 x 7 x 120 -> 720 -> 120 14.5 -> 10.2; batch 64 at width 1.0:
// 14 x 14 x 64 -> 384 -> 64 17.6 -> 13.7, but 56 x 56 x 24 -> 144 -> 24 44 -> 52.  Slices of 32 channels (an MMA of E reads its
// pixels twice as often, barriers and waits per unit count double) and 8 epilogue warps with two CTAs per SM were no
// faster anywhere.
#pragma once

#include "tc.cuh"

namespace prom { namespace block {

constexpr int kFirstEpi = 4;
constexpr int kSlice = 64;                          // expanded channels of a slice: bytes of a pixel in shared memory
constexpr int kHalf = 32;                           // ... of an MMA's K step and of a depthwise accumulator
constexpr uint32_t kUnitBytes = 128 * kSlice;       // an operand block of 128 pixels
constexpr uint32_t kStepBytes = 128 * kHalf;        // 128 input pixels x 32 channels
constexpr uint32_t kTapBytes = kHalf * kHalf;       // B of one depthwise tap of half a slice
constexpr uint32_t kHalfTaps = 10 * kTapBytes;      // ... of all nine, and the bias digits
constexpr int kRing = 8;                            // barriers of a kind
constexpr int kMaxCluster = 8;
constexpr int kEpiWarps = 16, kGroups = kEpiWarps / 4, kEpiThreads = 32 * kEpiWarps;
constexpr int kThreads = 32 * (kFirstEpi + kEpiWarps);

// A slice's prepared operands: expand weights (ks blocks of 64 rows x 32), bias digits (64 x 32), for each half
// nine depthwise taps (32 x 32) and bias digits, project weights (npad rows x 64), then constants as 32-bit
// words: four of a header {shift of E, or -1: any_constants; the same of D; halves with channels; whether a constant of E or D
// is out of range} and per channel as below (biases times four where any_constants takes them so).
enum { kMultE = 4, kMultD = kMultE + kSlice, kUpD = kMultD + kSlice, kBiasE = kUpD + kSlice, kBiasD = kBiasE + kSlice,
       kShiftE = kBiasD + kSlice, kShiftD = kShiftE + kSlice, kConstWords = kShiftD + kSlice };
constexpr int kToBias = kBiasE - kMultE, kToShift = kShiftE - kMultE;      // (the same for E and D)
static_assert(kToBias == kBiasD - kMultD && kToShift == kShiftD - kMultD, "one way from a multiplier to its bias and shift");
__host__ __device__ constexpr uint32_t off_taps(int ks) { return (uint32_t)(ks + 1) * 2 * kTapBytes; }
__host__ __device__ constexpr uint32_t off_project(int ks) { return off_taps(ks) + 2 * kHalfTaps; }
__host__ __device__ constexpr uint32_t off_consts(int ks, int npad) { return off_project(ks) + (uint32_t)npad * kSlice; }
// (whole swizzle atoms of 8 rows, so that a slot of the ring starts on one)
__host__ __device__ constexpr uint32_t slice_bytes(int ks, int npad) { return (off_consts(ks, npad) + 4 * kConstWords + 511u) & ~511u; }

enum { kBarWFull, kBarWEmpty, kBarXFull, kBarXEmpty, kBarD1Full, kBarD1Empty, kBarD2Full, kBarD2Empty, kBarEFull,
       kBarEEmpty, kBarPFull, kBarPEmpty, kBarD3Full, kBarD3Empty, kBarDrain, kBarKinds };
constexpr uint32_t kBarBytes = kBarKinds * kRing * 8;

constexpr uint32_t kNoPixel = 0xFFFFFFFFu;

struct Params {
    int batch, h, w, ho, wo, stride;
    int c0, co, npad;               // input and output channels; output channels rounded up to 16
    int rows, rin, bands, ipi;      // output rows of an item, its input rows, items per image, images per item
    int items, clusters;            // items in all, clusters (or CTAs) that take them in turn
    int pitch, qlen, plane;         // pixel buffer: pitch of a row, of an image, of a plane (stride 2)
    int t1, t2;                     // 128-pixel units of an item: expanded, output
    int ks;                         // K steps of 32 input channels
    int slices, per_cta, csize;     // slices of the layer and per CTA, CTAs of a cluster
    int n1, n2, np, ne;             // buffers (powers of two): accumulators of E and of D, operand blocks, pixel buffers
    int ns, nx;                     // ... of slices and of input pixels
    int ahead;                      // slices that E is in front of D: one less than the pixel buffers, at least 1
    int chunks;                     // an item's outputs in pieces of 128 pixels x 32 channels: t2 times the pieces of a pixel
    int tmem_cols, d2_col, d3_col;
    int tap[9];                     // byte offsets of the taps in the pixel buffer, in units of 16
    int px;                         // pieces of an input row: 16 bytes, or 8 where c0 is 8 modulo 16
    uint32_t px_magic;              // ceil(2^32 / px), for px above 1
    int last_half;                  // the last slice has channels in its first half only
    uint32_t per_img_magic, w_magic, qlen_magic, pitch_magic;      // ceil(2^32 / d) of rin * w, w, qlen and pitch
    int rpc, xpitch;                // cluster exchange: rows of a CTA, words of a row
    uint32_t slice_bytes, x_bytes, e_bytes;
    uint32_t off_e, off_p, off_w, off_aconst, off_etab, off_otab, off_pc, off_bars;
    const int8_t *x, *res;
    int8_t *y;
    const uint8_t *image;
    const int32_t *bias, *mult;     // of the project layer
    const int8_t *shift;
    int lo_e, hi_e, lo_d, hi_d, lo_p, hi_p;
    int pdl;
};

// ---- device helpers -----------------------------------------------------------------------------
// 32 accumulator columns of one pixel, clamp [0, 127], bias in the sum: the high word of a 64-bit
// multiply-add (rounding term in the addend), one shift, saturating pack, halve.  UP: the sums are first
// brought to the slice's common shift by a power of two per channel.
template <bool UP>
__device__ __forceinline__ void requant_32(const uint32_t (&v)[32], uint32_t mult, uint32_t up, int sh, uint32_t (&out)[8])
{
    const long long r64 = 1ll << (32 + sh);
#pragma unroll
    for (int c = 0; c < 32; c += 4) {
        const int4 mu = ptx::lds_128(mult + 4 * c);
        int t0 = (int)v[c], t1 = (int)v[c + 1], t2 = (int)v[c + 2], t3 = (int)v[c + 3];
        if constexpr (UP) {
            const int4 u = ptx::lds_128(up + 4 * c);
            t0 *= u.x; t1 *= u.y; t2 *= u.z; t3 *= u.w;
        }
        const int q0 = (int)(((long long)t0 * mu.x + r64) >> 32) >> sh, q1 = (int)(((long long)t1 * mu.y + r64) >> 32) >> sh;
        const int q2 = (int)(((long long)t2 * mu.z + r64) >> 32) >> sh, q3 = (int)(((long long)t3 * mu.w + r64) >> 32) >> sh;
        out[c / 4] = (ptx::pack_sat_u8(q1, q0, ptx::pack_sat_u8(q3, q2, 0u)) >> 1) & 0x7F7F7F7Fu;
    }
}

// A whole slice of one pixel with constants or clamps that requant_32 does not take.  Clamp [0, 127]: requant_floor with the
// bias (times four) and shift of every channel, 7 instructions per output against 4 (E) and 5 (D): slices in which a channel
// lies far from the others, a batch normalisation that has all but switched it off, say.  Any other clamp: the 64-bit definition.
// (A function of its own: inlined, bodies of the network whose constants do not need it took 2 % longer at batch 9, since the
// kernel's loops wait for their instructions.)
__device__ __noinline__ void any_constants(uint32_t taddr, const int *mult, int lo, int hi, int halves, uint32_t at, uint32_t swz, bool store, bool zero)
{
    if (lo == 0 && hi == 127) {
#pragma unroll 1
        for (int h = 0; h < halves; ++h) {
            uint32_t v[32], out[8];
            ptx::tmem_ld_x32(taddr + h * kHalf, v);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                const uint32_t o = ptx::smem_u32(mult + h * kHalf + c);
                const int4 mu = ptx::lds_128(o), bi = ptx::lds_128(o + 4 * kToBias), sh = ptx::lds_128(o + 4 * kToShift);
                const int q0 = (__mulhi((int)(4u * v[c]) + bi.x, mu.x) >> sh.x) + 1, q1 = (__mulhi((int)(4u * v[c + 1]) + bi.y, mu.y) >> sh.y) + 1;
                const int q2 = (__mulhi((int)(4u * v[c + 2]) + bi.z, mu.z) >> sh.z) + 1, q3 = (__mulhi((int)(4u * v[c + 3]) + bi.w, mu.w) >> sh.w) + 1;
                out[c / 4] = zero ? 0u : (ptx::pack_sat_u8(q1, q0, ptx::pack_sat_u8(q3, q2, 0u)) >> 1) & 0x7F7F7F7Fu;
            }
            if (store) {
                ptx::sts_128(at + ((32u * h) ^ swz), out[0], out[1], out[2], out[3]);
                ptx::sts_128(at + ((32u * h + 16u) ^ swz), out[4], out[5], out[6], out[7]);
            }
            __syncwarp();
        }
        return;
    }
    for (int h = 0; h < kSlice / 16; ++h) {
        uint32_t v[16];
        ptx::tmem_ld_x16(taddr + 16 * h, v);
        ptx::tmem_wait_ld();
        uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int c = 16 * h + i;
            const int q = zero ? 0 : requant_exact((int)v[i] + mult[kToBias + c], mult[c], mult[kToShift + c], lo, hi);
            o[i >> 2] |= ((uint32_t)q & 0xFFu) << (8 * (i & 3));
        }
        if (store) ptx::sts_128(at + (((uint32_t)h << 4) ^ swz), o[0], o[1], o[2], o[3]);
    }
}

// The project layer's constants in shared memory: mult, bias, power of two that brings the sum to the common
// shift, shift; npad each.  common: that shift (at least 2), or 0 where a channel cannot be brought to it.
struct Project {
    const int *c;
    int npad, common, lo, hi;
};
__device__ __noinline__ int project_exact(int acc, const int *c, int npad) { return requant_exact(acc + c[npad], c[0], c[3 * npad], -128, 127); }
// Eight outputs from channel c on.  Ties away from zero: the rounding term loses one unit where the product
// is negative, and its low word is empty, so the unit is the sign in both words.
__device__ __forceinline__ uint2 project_8(const Project &p, const int (&acc)[8], int c)
{
    int q[8];
    if (p.common) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t at = ptx::smem_u32(p.c + c + 4 * h);
            const int4 mu = ptx::lds_128(at), bi = ptx::lds_128(at + 4 * p.npad), up = ptx::lds_128(at + 8 * p.npad);
            const int m[4] = {mu.x, mu.y, mu.z, mu.w}, b[4] = {bi.x, bi.y, bi.z, bi.w}, u[4] = {up.x, up.y, up.z, up.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = (acc[4 * h + i] + b[i]) * u[i], sign = t >> 31;
                const unsigned long long add = ptx::pack_2((uint32_t)sign, (uint32_t)((1 << (p.common - 2)) + sign));
                q[4 * h + i] = (int)(((long long)t * m[i] + (long long)add) >> 32) >> (p.common - 1);
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            q[i] = project_exact(acc[i], p.c + c + i, p.npad);
    }
    if (p.lo != -128 || p.hi != 127) {
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = min(max(q[i], p.lo), p.hi);
    }
    return make_uint2(ptx::pack_sat_s8(q[1], q[0], ptx::pack_sat_s8(q[3], q[2], 0u)),
                      ptx::pack_sat_s8(q[5], q[4], ptx::pack_sat_s8(q[7], q[6], 0u)));
}

// What an item is.
struct Item {
    int img, y0, ys;                // first image, first output row, input row of the buffer's row 0
};
__device__ __forceinline__ Item item_of(const Params &p, int it)
{
    const int g = it / p.bands, b = it - g * p.bands;
    Item r;
    r.img = g * p.ipi; r.y0 = b * p.rows; r.ys = r.y0 * p.stride - 1;
    return r;
}

// Pieces [tid, tid + n, ..) below `end` of an item's input pixels into x buffer `dst`; the copies are asynchronous.
__device__ __forceinline__ void load_pixels(const Params &p, const Item &it, uint32_t dst, const uint32_t *etab, int tid, int n, int end)
{
    const int per_img = p.rin * p.w;
    const bool wide = (p.c0 & 15) == 0;
    const int8_t *origin = p.x + ((long long)it.img * p.h + it.ys) * p.w * p.c0;
    const int img_step = (p.h * p.w - per_img) * p.c0;              // (fits: the host sees to it)
#pragma unroll 4
    for (int i = tid; i < end; i += n) {
        const int m = p.px == 1 ? i : (int)__umulhi((uint32_t)i, p.px_magic), j = i - m * p.px;
        const uint32_t e = etab[m];
        const int r = (int)(e >> 16) & 0xFF, q = (int)(e >> 24), y = it.ys + r;
        const uint32_t b = (uint32_t)(wide ? 16 * j : 8 * j), row = (uint32_t)m & 127u;
        const int8_t *src = origin + (q * img_step + m * p.c0 + (int)b);
        const uint32_t d = dst + ((uint32_t)(m >> 7) * p.ks + (b >> 5)) * kStepBytes + tc::swz_offset(row, (b >> 4) & 1u, 32u) + (b & 15u);
        if ((unsigned)y < (unsigned)p.h && it.img + q < p.batch) {
            if (wide) ptx::cp_async_16(d, src);
            else ptx::cp_async_8(d, src);
        }
    }
}

// n / d for n below 2^14 with magic = ceil(2^32 / d), d above 1.
__device__ __forceinline__ int div_by(int n, uint32_t magic) { return (int)__umulhi((uint32_t)n, magic); }

// A position in a ring: index and phase.
struct Ring {
    uint32_t i = 0, ph = 0;
    __device__ __forceinline__ void next(int n) { if (++i == (uint32_t)n) { i = 0; ph ^= 1u; } }
};
// A count as a position in the rings of eight barriers.
__device__ __forceinline__ uint32_t at8(uint32_t n) { return n & (kRing - 1); }
__device__ __forceinline__ uint32_t phase8(uint32_t n) { return (n / kRing) & 1u; }

__global__ void __launch_bounds__(kThreads, 1) block_kernel(const __grid_constant__ Params p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t base = ptx::smem_u32(smem);
    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + p.off_bars);
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto bar = [&](int kind, uint32_t i) { return bar0 + 8u * (uint32_t)(kind * kRing) + 8u * i; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + p.off_bars + kBarBytes);
    volatile int *flags = reinterpret_cast<volatile int *>(smem + p.off_bars + kBarBytes) + 2;     // [0] abort
    int *pspan = reinterpret_cast<int *>(smem + p.off_bars + kBarBytes) + 4;     // project layer: smallest shift (-1: a constant of
                                                                                 // the block is out of range), largest, largest |bias|
    uint32_t *etab = reinterpret_cast<uint32_t *>(smem + p.off_etab), *otab = reinterpret_cast<uint32_t *>(smem + p.off_otab);
    int *pc = reinterpret_cast<int *>(smem + p.off_pc);

    const int rank = p.csize > 1 ? (int)ptx::cluster_rank() : 0;
    const int cluster = blockIdx.x / p.csize;
    const int s_first = rank * p.per_cta;
    const int nsl = min(p.per_cta, p.slices - s_first);            // at least one: the host sees to it
    const int n_items = (p.items - cluster + p.clusters - 1) / p.clusters;
    const int total = n_items * nsl;

    if (p.pdl != tc::kPdlWait) ptx::grid_dep_launch();
    if (warp == 0) {
        if (lane < kRing) {
            const uint32_t i = (uint32_t)lane;
            ptx::mbar_init(bar(kBarWFull, i), 1); ptx::mbar_init(bar(kBarWEmpty, i), 1);
            ptx::mbar_init(bar(kBarXFull, i), kEpiWarps); ptx::mbar_init(bar(kBarXEmpty, i), 1);
            ptx::mbar_init(bar(kBarD1Full, i), 1); ptx::mbar_init(bar(kBarD1Empty, i), 4);
            ptx::mbar_init(bar(kBarD2Full, i), 1); ptx::mbar_init(bar(kBarD2Empty, i), 4);
            ptx::mbar_init(bar(kBarEFull, i), 4 * p.t1); ptx::mbar_init(bar(kBarEEmpty, i), 1);
            ptx::mbar_init(bar(kBarPFull, i), 4); ptx::mbar_init(bar(kBarPEmpty, i), 1);
            ptx::mbar_init(bar(kBarD3Full, i), 2); ptx::mbar_init(bar(kBarD3Empty, i), 4 * p.chunks);
            ptx::mbar_init(bar(kBarDrain, i), 1);
        }
        if (lane == 0) flags[0] = 0;
        ptx::mbar_init_fence();
        __syncwarp();
    }
    if (p.pdl == tc::kPdlWait) {
        ptx::grid_dep_wait();
        ptx::grid_dep_launch();
    }
    // the slices' operands do not depend on the kernel in front: the first ones are asked for at once
    auto load_slice = [&](uint32_t slot, int s) {
        ptx::mbar_expect_tx(bar(kBarWFull, slot), p.slice_bytes);
        ptx::bulk_load(base + p.off_w + slot * p.slice_bytes, p.image + (size_t)(s_first + s) * p.slice_bytes, p.slice_bytes,
                       bar(kBarWFull, slot));
    };
    const int pre = min(p.ns, total);
    if (warp == 0 && lane == 0)
        for (int i = 0, s = 0; i < pre; ++i) {
            load_slice((uint32_t)i, s);
            if (++s == nsl) s = 0;
        }
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32((const void *)tmem_slot), (uint32_t)p.tmem_cols);
    {
        // where an expanded pixel goes in the pixel buffer, and which output a lane of D and P is
        const int per_img = p.rin * p.w;
        for (int m = threadIdx.x; m < 128 * p.t1; m += kThreads) {
            const int q = div_by(m, p.per_img_magic), mm = m - q * per_img, r = p.w == 1 ? mm : div_by(mm, p.w_magic), c = mm - r * p.w + 1;
            const int idx = p.stride == 1 ? q * p.qlen + r * p.pitch + c
                                          : ((r & 1) * 2 + (c & 1)) * p.plane + q * p.qlen + (r >> 1) * p.pitch + (c >> 1);
            etab[m] = q < p.ipi ? (uint32_t)idx | ((uint32_t)r << 16) | ((uint32_t)q << 24) : kNoPixel;
        }
        for (int i = threadIdx.x; i < 128 * p.t2; i += kThreads) {
            const int q = div_by(i, p.qlen_magic), ii = i - q * p.qlen, oy = div_by(ii, p.pitch_magic), ox = ii - oy * p.pitch;
            otab[i] = q < p.ipi && oy < p.rows && ox < p.wo ? (uint32_t)(oy * p.wo + ox) | ((uint32_t)oy << 16) | ((uint32_t)q << 24)
                                                            : kNoPixel;
        }
        for (uint32_t i = threadIdx.x; i < (uint32_t)p.ne * p.e_bytes / 16; i += kThreads)
            ptx::sts_128(base + p.off_e + 16 * i, 0u, 0u, 0u, 0u);
        tc::build_aconst(smem + p.off_aconst, (int)threadIdx.x, kThreads);
        if (threadIdx.x == 64) { pspan[0] = 31; pspan[1] = 0; pspan[2] = 0; }
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // s8 x s8 -> s32, both K-major, M = 128
    constexpr uint32_t kI0 = (2u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
    constexpr uint32_t kI32 = kI0 | ((uint32_t)(kHalf >> 3) << 17), kI64 = kI0 | ((uint32_t)(kSlice >> 3) << 17);
    const uint64_t d32 = tc::smem_desc(0u, 32u), d64 = tc::smem_desc(0u, 64u);
    const uint64_t ac = d32 | (uint64_t)((base + p.off_aconst) >> 4);
    const uint32_t w_lo = (base + p.off_w) >> 4, w_step = p.slice_bytes >> 4;
    bool ok = true;

    if (warp == 0) {
        // ---- slices and, from the second item on (the epilogue warps load the first one's), input pixels -------
        // Whichever has room; pixels a few at a time, so that a slice does not wait for them.
        if (p.pdl == tc::kPdlChain) ptx::grid_dep_wait();
        const bool leader = ptx::elect_one();
        const int pieces = p.ipi * p.rin * p.w * p.px;
        int issued = pre, s = pre % nsl, j = 1, at = -1;        // at: pieces of item j on their way, or -1: its buffer is in use
        Ring w, x;
        for (int i = 0; i < pre; ++i) w.next(p.ns);
        x.next(p.nx);
        unsigned long long t0 = 0;
        for (uint32_t polls = 1; issued < total || j < n_items; ++polls) {
            if (issued < total && __all_sync(0xFFFFFFFFu, ptx::mbar_test_wait(bar(kBarWEmpty, w.i), w.ph ^ 1u))) {
                if (leader) load_slice(w.i, s);
                w.next(p.ns);
                if (++s == nsl) s = 0;
                ++issued;
                t0 = 0; polls = 0;
            }
            if (j < n_items) {
                if (at < 0 && __all_sync(0xFFFFFFFFu, ptx::mbar_test_wait(bar(kBarXEmpty, x.i), x.ph ^ 1u))) at = 0;
                if (at >= 0) {
                    const int end = min(at + 32 * 8, pieces);
                    load_pixels(p, item_of(p, cluster + j * p.clusters), base + x.i * p.x_bytes, etab, at + lane, 32, end);
                    at = end;
                    if (at == pieces) {
                        ptx::cp_async_wait_all();
                        ptx::fence_proxy_async_smem();
                        __syncwarp();
                        if (leader) ptx::mbar_arrive_n(bar(kBarXFull, x.i), kEpiWarps);
                        x.next(p.nx);
                        ++j; at = -1;
                    }
                    t0 = 0; polls = 0;
                }
            }
            if ((polls & 1023u) == 1023u) {
                t0 = tc::wait_check(t0, flags, tc::kWaitLimitNs);
                if (__any_sync(0xFFFFFFFFu, t0 == tc::kWaitGiveUp)) { ok = false; break; }
            }
        }
        ptx::cp_async_wait_all();
        if (leader) tc::drain_copies(bar(kBarWFull, 0), (uint32_t)p.ns, (uint32_t)issued);
        __syncwarp();
    } else if (warp == 1) {
        // ---- E ----------------------------------------------------------------------------------------
        const bool leader = ptx::elect_one();
        Ring w, x;
        uint32_t u = 0;
        for (int j = 0; j < n_items && ok; ++j) {
            if (!tc::wait_bar_warp(bar(kBarXFull, x.i), x.ph, flags)) { ok = false; break; }
            const uint32_t xa = (base + x.i * p.x_bytes) >> 4;
            for (int s = 0; s < nsl && ok; ++s) {
                const uint32_t idesc = p.last_half && s_first + s == p.slices - 1 ? kI32 : kI64;
                if (!tc::wait_bar_warp(bar(kBarWFull, w.i), w.ph, flags)) { ok = false; break; }
                const uint32_t b = w_lo + w.i * w_step;
                uint32_t a = xa;
                for (int t = 0; t < p.t1; ++t, ++u) {
                    const uint32_t o = u - (uint32_t)p.n1;          // the accumulator's unit before
                    if (u >= (uint32_t)p.n1 && !tc::wait_bar_warp(bar(kBarD1Empty, at8(o)), phase8(o), flags)) { ok = false; break; }
                    ptx::tc_fence_after_sync();
                    const uint32_t dst = tmem + (u & (uint32_t)(p.n1 - 1)) * kSlice;
                    if (leader) {
                        ptx::mma_i8<false>(dst, ac, d32 | (uint64_t)(b + (uint32_t)p.ks * (2 * kTapBytes >> 4)), idesc);
                        for (int k = 0; k < p.ks; ++k)
                            ptx::mma_i8<true>(dst, d32 | (uint64_t)(a + (uint32_t)k * (kStepBytes >> 4)),
                                              d32 | (uint64_t)(b + (uint32_t)k * (2 * kTapBytes >> 4)), idesc);
                        ptx::mma_commit(bar(kBarD1Full, at8(u)));
                    }
                    a += (uint32_t)p.ks * (kStepBytes >> 4);
                }
                w.next(p.ns);
            }
            if (leader) ptx::mma_commit(bar(kBarXEmpty, x.i));
            x.next(p.nx);
        }
    } else if (warp == 2) {
        // ---- D ----------------------------------------------------------------------------------------
        const bool leader = ptx::elect_one();
        Ring w;
        uint32_t v = 0;
        int s = 0;
        for (int k = 0; k < total && ok; ++k) {
            const int halves = p.last_half && s_first + s == p.slices - 1 ? 1 : 2;
            if (++s == nsl) s = 0;
            if (!tc::wait_bar_warp(bar(kBarWFull, w.i), w.ph, flags) ||
                !tc::wait_bar_warp(bar(kBarEFull, at8((uint32_t)k)), phase8((uint32_t)k), flags)) {
                ok = false;
                break;
            }
            const uint32_t b = w_lo + w.i * w_step + (off_taps(p.ks) >> 4);
            uint32_t a = (base + p.off_e + ((uint32_t)k & (uint32_t)(p.ne - 1)) * p.e_bytes) >> 4;
            for (int t = 0; t < p.t2; ++t, ++v) {
                const uint32_t o = v - (uint32_t)p.n2;
                if (v >= (uint32_t)p.n2 && !tc::wait_bar_warp(bar(kBarD2Empty, at8(o)), phase8(o), flags)) { ok = false; break; }
                ptx::tc_fence_after_sync();
                uint32_t dst = tmem + (uint32_t)p.d2_col + (v & (uint32_t)(p.n2 - 1)) * kSlice;
                if (leader) {
                    uint32_t bh = b, ah = a;
                    for (int h = 0; h < halves; ++h) {
                        ptx::mma_i8<false>(dst, ac, d32 | (uint64_t)(bh + 9 * (kTapBytes >> 4)), kI32);
#pragma unroll
                        for (int i = 0; i < 9; ++i)
                            ptx::mma_i8<true>(dst, d64 | (uint64_t)(ah + (uint32_t)p.tap[i]), d32 | (uint64_t)(bh + i * (kTapBytes >> 4)), kI32);
                        bh += kHalfTaps >> 4; ah += kHalf >> 4; dst += kHalf;
                    }
                    ptx::mma_commit(bar(kBarD2Full, at8(v)));
                }
                a += kUnitBytes >> 4;
            }
            if (leader) ptx::mma_commit(bar(kBarEEmpty, at8((uint32_t)k)));
            w.next(p.ns);
        }
    } else if (warp == 3) {
        // ---- P ----------------------------------------------------------------------------------------
        const bool leader = ptx::elect_one();
        Ring w;
        uint32_t v = 0;
        int bad = 0;
        const int n_a = min(p.npad, 256), n_b = p.npad - n_a;      // an MMA is at most 256 columns wide
        const uint32_t i_a = kI0 | ((uint32_t)(n_a >> 3) << 17), i_b = kI0 | ((uint32_t)(n_b >> 3) << 17);
        for (int j = 0; j < n_items && ok; ++j) {
            if (!tc::wait_bar_warp(bar(kBarD3Empty, 0), ((uint32_t)j & 1u) ^ 1u, flags)) { ok = false; break; }
            for (int s = 0; s < nsl && ok; ++s) {
                const bool two = !(p.last_half && s_first + s == p.slices - 1);
                if (!tc::wait_bar_warp(bar(kBarWFull, w.i), w.ph, flags)) { ok = false; break; }
                bad |= *reinterpret_cast<const volatile int *>(smem + p.off_w + w.i * p.slice_bytes + off_consts(p.ks, p.npad) + 12);
                const uint64_t b = d64 | (uint64_t)(w_lo + w.i * w_step + (off_project(p.ks) >> 4));
                for (int t = 0; t < p.t2; ++t, ++v) {
                    if (!tc::wait_bar_warp(bar(kBarPFull, at8(v)), phase8(v), flags)) { ok = false; break; }
                    ptx::tc_fence_after_sync();
                    const uint64_t a = d64 | (uint64_t)((base + p.off_p + (v & (uint32_t)(p.np - 1)) * kUnitBytes) >> 4);
                    const uint32_t dst = tmem + (uint32_t)(p.d3_col + t * p.npad);
                    if (leader) {
                        ptx::mma_i8(dst, a, b, i_a, s > 0);
                        if (two) ptx::mma_i8<true>(dst, a + (kHalf >> 4), b + (kHalf >> 4), i_a);
                        if (n_b) {
                            ptx::mma_i8(dst + 256, a, b + (256 * kSlice >> 4), i_b, s > 0);
                            if (two) ptx::mma_i8<true>(dst + 256, a + (kHalf >> 4), b + (256 * kSlice + kHalf >> 4), i_b);
                        }
                        ptx::mma_commit(bar(kBarPEmpty, at8(v)));
                    }
                }
                if (leader) ptx::mma_commit(bar(kBarWEmpty, w.i));
                w.next(p.ns);
            }
            if (leader) {
                if (bad) atomicMin(pspan, -1);
                ptx::mbar_arrive(bar(kBarD3Full, 0));
                ptx::mma_commit(bar(kBarD3Full, 0));
            }
        }
    } else {
        // ---- epilogue -----------------------------------------------------------------------------------
        const int etid = (int)threadIdx.x - 32 * kFirstEpi, grp = (warp - kFirstEpi) >> 2, quarter = warp & 3;
        const uint32_t t_lane = tmem + ((uint32_t)(quarter * 32) << 16);
        if (p.pdl == tc::kPdlChain) ptx::grid_dep_wait();
        load_pixels(p, item_of(p, cluster), base, etab, etid, kEpiThreads, p.ipi * p.rin * p.w * p.px);
        // beside those loads, the project layer's constants.  Common shift: |sum| <= 4096 * 128 plus the bias, times
        // 2^10, stays within 31 bits for a bias below 2^20
        // (a constant out of range: a smallest shift of -1, and no output is written)
        int mn = 31, mx = 0, ab = 0;
        for (int c = etid; c < p.npad; c += kEpiThreads) {
            int b = 0, mu = 0, sh = -1;
            if (c < p.co) {
                b = __ldg(p.bias + c); mu = __ldg(p.mult + c); sh = __ldg(p.shift + c);
                if (!requant_ok(b, mu, sh)) { raise_status(PROM_ERR_BAD_REQUANT); b = 0; mu = 0; sh = 0; mn = -1; }
                mn = min(mn, sh); mx = max(mx, sh); ab = max(ab, abs(b));
            }
            pc[c] = mu; pc[p.npad + c] = b; pc[3 * p.npad + c] = sh;
        }
        ptx::cp_async_wait_all();
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar(kBarXFull, 0));
        {
            mn = __reduce_min_sync(0xFFFFFFFFu, mn); mx = __reduce_max_sync(0xFFFFFFFFu, mx); ab = __reduce_max_sync(0xFFFFFFFFu, ab);
            if (lane == 0 && 32 * (warp - kFirstEpi) < p.co) { atomicMin(pspan, mn); atomicMax(pspan + 1, mx); atomicMax(pspan + 2, ab); }
            ptx::named_sync(1, kEpiThreads);
            const int top = max(pspan[1], 2);
            for (int c = etid; c < p.npad; c += kEpiThreads) {
                const int sh = pc[3 * p.npad + c];
                pc[2 * p.npad + c] = sh >= 0 && top - sh <= 10 ? 1 << (top - sh) : 0;
            }
            ptx::named_sync(1, kEpiThreads);
        }
        const int top = max(pspan[1], 2);
        const Project prj = {pc, p.npad, top - pspan[0] <= 10 && pspan[2] < (1 << 20) ? top : 0, p.lo_p, p.hi_p};
        auto wait = [&](uint32_t b, uint32_t ph) { return __all_sync(0xFFFFFFFFu, tc::wait_bar(b, ph, flags)); };
        auto wait_2 = [&](uint32_t b1, uint32_t p1, uint32_t b2, uint32_t p2) {
            return __all_sync(0xFFFFFFFFu, tc::wait_bar(b1, p1, flags) && tc::wait_bar(b2, p2, flags));
        };

        // an item's outputs, from the sums in tensor memory (no cluster): 32 channels of a pixel at a time
        const int per_px = p.chunks / p.t2;
        auto finish = [&](int j) {
            const Item it = item_of(p, cluster + j * p.clusters);
            bool waited = false;
            for (int i = grp; i < p.chunks; i += kGroups) {
                const int t = i / per_px, c0 = 32 * (i - t * per_px);
                const uint32_t o = otab[128 * t + 32 * quarter + lane];
                const int oy = (int)(o >> 16) & 0xFF, q = (int)(o >> 24);
                const bool valid = o != kNoPixel && it.y0 + oy < p.ho && it.img + q < p.batch;
                const long long at = ((long long)((it.img + q) * p.ho + it.y0) * p.wo + (int)(o & 0xFFFFu)) * p.co + c0;
                const bool add = p.res != nullptr && valid;
                uint2 r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    r[e] = add && c0 + 8 * e < p.co ? __ldcg(reinterpret_cast<const uint2 *>(p.res + at + 8 * e)) : make_uint2(0u, 0u);
                if (!waited) {
                    if (!wait(bar(kBarD3Full, 0), (uint32_t)j & 1u)) return false;
                    ptx::tc_fence_after_sync();
                    waited = true;
                }
                __syncwarp();
                const bool write = valid && *reinterpret_cast<volatile int *>(pspan) >= 0;
                const uint32_t sums = t_lane + (uint32_t)(p.d3_col + t * p.npad + c0);
                const int n = min(p.co - c0, 32);
                // (rolled: straight-line code for a few outputs per thread waits for its instructions)
#pragma unroll 1
                for (int e = 0; e < n; e += 8) {
                    uint32_t z[8];
                    ptx::tmem_ld_x8(sums + e, z);
                    ptx::tmem_wait_ld();
                    const int a[8] = {(int)z[0], (int)z[1], (int)z[2], (int)z[3], (int)z[4], (int)z[5], (int)z[6], (int)z[7]};
                    uint2 out = project_8(prj, a, c0 + e);
                    if (add) { out.x = __vaddss4(out.x, r[0].x); out.y = __vaddss4(out.y, r[0].y); }
                    if (write) *reinterpret_cast<uint2 *>(p.y + at + e) = out;
                    r[0] = r[1]; r[1] = r[2]; r[2] = r[3];
                    __syncwarp();
                }
                tc::release_acc(bar(kBarD3Empty, 0));
            }
            return true;
        };

        Ring we, wd;                            // slices of E and of D
        int te = grp, td = (grp + kGroups / 2) % kGroups;      // this group's next unit, counted from its slice's first
        int se = 0, sd = 0, je = 0, jd = 0;     // slice and item of E and of D
        uint32_t u0 = 0, v0 = 0;                // units of E and of D in the slices before
        int ys = item_of(p, cluster).ys;
        const uint32_t consts = p.off_w + off_consts(p.ks, p.npad);
        const uint32_t my_row = (uint32_t)(32 * quarter + lane);
        auto expand = [&](int k) {               // this group's next unit of E, of slice k
            const uint32_t u = u0 + (uint32_t)te, off_c = consts + we.i * p.slice_bytes;
            const uint32_t px = etab[128u * te + my_row];
            const bool store = px != kNoPixel;
            const bool zero = (unsigned)(ys + (int)((px >> 16) & 0xFFu)) >= (unsigned)p.h;
            const uint32_t at = base + p.off_e + ((uint32_t)k & (uint32_t)(p.ne - 1)) * p.e_bytes + (px & 0xFFFFu) * kSlice;
            const uint32_t swz = ((at >> 7) & 3u) << 4;
            const uint32_t acc = t_lane + (u & (uint32_t)(p.n1 - 1)) * kSlice;
            const uint32_t o = (uint32_t)(k - p.ne);                 // the pixel buffer's slice before
            ok = k >= p.ne ? wait_2(bar(kBarEEmpty, at8(o)), phase8(o), bar(kBarD1Full, at8(u)), phase8(u))
                           : wait(bar(kBarD1Full, at8(u)), phase8(u));
            if (!ok) return;
            ptx::tc_fence_after_sync();
            const int4 hdr = ptx::lds_128(base + off_c);
            if (hdr.x >= 0) {
#pragma unroll 1
                for (int h = 0; h < hdr.z; ++h) {
                    uint32_t acc_v[32], out[8];
                    ptx::tmem_ld_x32(acc + h * kHalf, acc_v);
                    ptx::tmem_wait_ld();
                    if (h + 1 == hdr.z) tc::release_acc(bar(kBarD1Empty, at8(u)));
                    requant_32<false>(acc_v, base + off_c + 4 * (kMultE + h * kHalf), 0u, hdr.x, out);
                    if (zero) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) out[i] = 0u;
                    }
                    if (store) {
                        ptx::sts_128(at + ((32u * h) ^ swz), out[0], out[1], out[2], out[3]);
                        ptx::sts_128(at + ((32u * h + 16u) ^ swz), out[4], out[5], out[6], out[7]);
                    }
                    __syncwarp();
                }
            } else {
                any_constants(acc, reinterpret_cast<const int *>(smem + off_c) + kMultE, p.lo_e, p.hi_e, hdr.z, at, swz, store, zero);
                tc::release_acc(bar(kBarD1Empty, at8(u)));
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(kBarEFull, at8((uint32_t)k)));
            te += kGroups;
        };
        auto depthwise = [&]() {                 // ... of D
            const uint32_t v = v0 + (uint32_t)td, off_c = consts + wd.i * p.slice_bytes;
            const uint32_t at = base + p.off_p + (v & (uint32_t)(p.np - 1)) * kUnitBytes + my_row * kSlice;
            const uint32_t swz = ((at >> 7) & 3u) << 4, acc = t_lane + (uint32_t)p.d2_col + (v & (uint32_t)(p.n2 - 1)) * kSlice;
            const uint32_t o = v - (uint32_t)p.np;                       // the operand block's unit before
            ok = v >= (uint32_t)p.np ? wait_2(bar(kBarPEmpty, at8(o)), phase8(o), bar(kBarD2Full, at8(v)), phase8(v))
                                     : wait(bar(kBarD2Full, at8(v)), phase8(v));
            if (!ok) return;
            ptx::tc_fence_after_sync();
            const int4 hdr = ptx::lds_128(base + off_c);
            if (hdr.y >= 0) {
#pragma unroll 1
                for (int h = 0; h < hdr.z; ++h) {
                    uint32_t acc_v[32], out[8];
                    ptx::tmem_ld_x32(acc + h * kHalf, acc_v);
                    ptx::tmem_wait_ld();
                    if (h + 1 == hdr.z) tc::release_acc(bar(kBarD2Empty, at8(v)));
                    requant_32<true>(acc_v, base + off_c + 4 * (kMultD + h * kHalf), base + off_c + 4 * (kUpD + h * kHalf), hdr.y, out);
                    ptx::sts_128(at + ((32u * h) ^ swz), out[0], out[1], out[2], out[3]);
                    ptx::sts_128(at + ((32u * h + 16u) ^ swz), out[4], out[5], out[6], out[7]);
                }
            } else {
                any_constants(acc, reinterpret_cast<const int *>(smem + off_c) + kMultD, p.lo_d, p.hi_d, hdr.z, at, swz, true, false);
                tc::release_acc(bar(kBarD2Empty, at8(v)));
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(kBarPFull, at8(v)));
            td += kGroups;
        };
        // All groups keep to one order of the units: half a turn of E, half a turn of D, and so on, E `ahead` slices in
        // front; so D's MMAs, most of the tensor pipe's work, run beside both.  An item's outputs come in front of the
        // next one's first units of D, behind a turn of E.
        constexpr int kHalfTurn = kGroups / 2;
        for (int k = 0; k < total + p.ahead && ok; ++k) {
            const int n_e = k < total ? p.t1 : 0, n_d = k >= p.ahead ? p.t2 : 0;
            if (n_d && sd == 0 && jd > 0) {
                if (te < n_e) expand(k);
                if (ok) ok = finish(jd - 1);
            }
            while (ok && (te < n_e || td < n_d)) {
                if (te < n_e && (td >= n_d || te / kHalfTurn <= td / kHalfTurn)) expand(k);
                else depthwise();
            }
            if (n_e) {
                te -= p.t1; u0 += (uint32_t)p.t1;
                we.next(p.ns);
                if (++se == nsl) {
                    se = 0;
                    ys = item_of(p, cluster + ++je * p.clusters).ys;
                }
            }
            if (n_d) {
                td -= p.t2; v0 += (uint32_t)p.t2;
                wd.next(p.ns);
                if (++sd == nsl) { sd = 0; ++jd; }
            }
        }
        if (ok && p.csize == 1) ok = finish(n_items - 1);
        if (ok && p.csize > 1) {
            ok = wait(bar(kBarD3Full, 0), 0u);          // (a cluster has one item)
            ptx::tc_fence_after_sync();
        }
    }
    // MMAs in flight when a role has given up end before tensor memory goes
    if (!ok && warp >= 1 && warp <= 3) {
        if (lane == 0) {
            ptx::mma_commit(bar(kBarDrain, (uint32_t)warp));
            const unsigned long long g0 = ptx::globaltimer();
            while (!ptx::mbar_try_wait(bar(kBarDrain, (uint32_t)warp), 0) && ptx::globaltimer() - g0 < tc::kWaitLimitNs) {}
        }
    }
    __syncwarp();

    if (p.csize > 1) {
        // A thread's sums go to the CTA that owns its pixel, 16 channels at a time, the groups in turn.  Where they go, and
        // the first of them, are found in front of the barrier behind which every CTA's MMAs have read what they need
        // and shared memory up to off_aconst holds sums.
        const Item it = item_of(p, cluster);
        const bool mine = warp >= kFirstEpi && ok;
        const int grp = (warp - kFirstEpi) >> 2;
        const uint32_t my_lane = (uint32_t)(32 * (warp & 3) + lane), t_sums = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)p.d3_col;
        uint32_t to = 0;
        bool valid = false;
        auto target = [&](int t) {
            const uint32_t o = otab[128u * t + my_lane];
            const int r = (int)(o >> 24) * p.rows * p.wo + (int)(o & 0xFFFFu);
            valid = o != kNoPixel;
            const int owner = valid ? r / p.rpc : 0;
            to = ptx::map_to_rank(base, (uint32_t)owner) + 4u * (uint32_t)((rank * p.rpc + r - owner * p.rpc) * p.xpitch);
        };
        uint32_t z[16];
        if (mine) {
            target(0);
            if (16 * grp < p.npad) {
                ptx::tmem_ld_x16(t_sums + 16 * grp, z);
                ptx::tmem_wait_ld();
            }
        }
        __syncwarp();
        ptx::cluster_sync();
        if (mine) {
#pragma unroll 1
            for (int t = 0; t < p.t2; ++t) {
                if (t) target(t);
#pragma unroll 1
                for (int c0 = 16 * grp; c0 < p.npad; c0 += 16 * kGroups) {
                    if (t || c0 != 16 * grp) {
                        ptx::tmem_ld_x16(t_sums + (uint32_t)(t * p.npad + c0), z);
                        ptx::tmem_wait_ld();
                    }
                    if (valid) {
#pragma unroll
                        for (int e = 0; e < 16; e += 8) {
                            if (c0 + e >= p.co) break;
                            ptx::st_cluster_v4(to + 4 * (c0 + e), z[e], z[e + 1], z[e + 2], z[e + 3]);
                            ptx::st_cluster_v4(to + 4 * (c0 + e) + 16, z[e + 4], z[e + 5], z[e + 6], z[e + 7]);
                        }
                    }
                    __syncwarp();
                }
            }
        }
        // (a constant out of range in one CTA's slices: no CTA writes)
        if (warp == 3 && lane < p.csize && pspan[0] < 0) ptx::st_cluster_32(ptx::map_to_rank(ptx::smem_u32(pspan), (uint32_t)lane), 0xFFFFFFFFu);
        // this thread's outputs: eight channels of pixel rr of the CTA's share, then every kEpiThreads-th such piece
        const int etid = (int)threadIdx.x - 32 * kFirstEpi, c8 = p.co >> 3, plane = p.rows * p.wo;
        const int share = min(p.rpc, p.ipi * plane - rank * p.rpc) * c8;
        auto place = [&](int i, int &rr, int &c) {
            rr = i / c8; c = 8 * (i - rr * c8);
            const int r = rank * p.rpc + rr, q = r / plane, in = r - q * plane;
            const bool there = it.y0 + in / p.wo < p.ho && it.img + q < p.batch;
            return there ? ((long long)((it.img + q) * p.ho + it.y0) * p.wo + in) * p.co + c : -1ll;
        };
        int rr = 0, c = 0;
        long long at = mine && etid < share ? place(etid, rr, c) : -1ll;
        uint2 rs = make_uint2(0u, 0u);
        if (p.res && at >= 0) rs = __ldcg(reinterpret_cast<const uint2 *>(p.res + at));
        __syncwarp();
        ptx::cluster_sync();
        if (mine) {
            const int top = max(pspan[1], 2);
            const Project prj = {pc, p.npad, top - pspan[0] <= 10 && pspan[2] < (1 << 20) ? top : 0, p.lo_p, p.hi_p};
            const bool write = pspan[0] >= 0;
            for (int i = etid; i < share; i += kEpiThreads) {
                if (i != etid) {
                    at = place(i, rr, c);
                    if (p.res && at >= 0) rs = __ldcg(reinterpret_cast<const uint2 *>(p.res + at));
                }
                if (at < 0) continue;
                int sum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                for (int k = 0; k < p.csize; ++k) {
                    const uint32_t src = base + 4u * (uint32_t)((k * p.rpc + rr) * p.xpitch + c);
                    const int4 a = ptx::lds_128(src), b = ptx::lds_128(src + 16);
                    sum[0] += a.x; sum[1] += a.y; sum[2] += a.z; sum[3] += a.w;
                    sum[4] += b.x; sum[5] += b.y; sum[6] += b.z; sum[7] += b.w;
                }
                uint2 out = project_8(prj, sum, c);
                if (p.res) { out.x = __vaddss4(out.x, rs.x); out.y = __vaddss4(out.y, rs.y); }
                if (write) *reinterpret_cast<uint2 *>(p.y + at) = out;
            }
        }
    }
    // ---- teardown -------------------------------------------------------------------------------------
    if (p.pdl == tc::kPdlChain && threadIdx.x == 32) ptx::grid_dep_wait();
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
    }
}

// ---- the slices' operands -----------------------------------------------------------------------------
struct PrepBlock {
    const uint8_t *we, *wp;                     // packed weights of the expand and the project layer
    const int32_t *bias_e, *mult_e, *bias_d, *mult_d;
    const int8_t *shift_e, *shift_d, *wd;
    uint8_t *image;
    int c0, ce, co, npad, ks;
    int lo_e, hi_e, lo_d, hi_d;
    int first;                                  // first CTA
};
constexpr int kMaxPrep = 24;
constexpr int kPrepThreads = 512;
struct PrepTable {
    int n;
    int behind;                                 // the kernel in front is this call's own and reads nothing written here
    PrepBlock b[kMaxPrep];
};

// One CTA per slice.
__global__ void __launch_bounds__(kPrepThreads) block_prep_kernel(const __grid_constant__ PrepTable t)
{
    __shared__ int cst[kConstWords];
    __shared__ int scale_e[kSlice];              // the expand weights are +-2^this
    __shared__ int span[7];
    const int tid = (int)threadIdx.x;
    int l = 0;
    while (l + 1 < t.n && (int)blockIdx.x >= t.b[l + 1].first) ++l;
    const PrepBlock &p = t.b[l];
    const int slice = (int)blockIdx.x - p.first, ch0 = slice * kSlice;
    uint8_t *const image = p.image + (size_t)slice * slice_bytes(p.ks, p.npad);
    if (!t.behind) ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    if (tid == 0) { span[0] = 31; span[1] = 0; span[2] = 0; span[3] = 2; span[4] = 0; span[5] = 31; span[6] = 0; }
    __syncthreads();
    int be = 0, me = 0, se = 0, bd = 0, md = 0, sd = 0;
    const bool mine = tid < kSlice && ch0 + tid < p.ce;
    if (tid < kSlice) {
        // constants, and whether the one-multiply epilogues apply (the conditions of tc.cuh and dwtc.cuh)
        const int ch = ch0 + tid;
        if (mine) {
            be = __ldg(p.bias_e + ch); me = __ldg(p.mult_e + ch); se = __ldg(p.shift_e + ch);
            bd = __ldg(p.bias_d + ch); md = __ldg(p.mult_d + ch); sd = __ldg(p.shift_d + ch);
            if (!requant_ok(be, me, se)) { raise_status(PROM_ERR_BAD_REQUANT); be = 0; me = 0; se = 0; span[6] = 1; }
            if (!requant_ok(bd, md, sd)) { raise_status(PROM_ERR_BAD_REQUANT); bd = 0; md = 0; sd = 0; span[6] = 1; }
            atomicMin(&span[0], se); atomicMax(&span[1], se);
            const long long ab = be < 0 ? -(long long)be : be;
            if ((((long long)128 * p.c0 + ab) << 6) >= (1ll << 31) || (ab << 6) > tc::kBiasMax) span[2] = 1;
            atomicMax(&span[3], sd); atomicMin(&span[5], sd);
            if (bd < -tc::kBiasMax || bd > tc::kBiasMax) span[4] = 1;
        }
    }
    __syncthreads();
    if (tid < kSlice) {
        const bool relu_e = p.lo_e == 0 && p.hi_e == 127, relu_d = p.lo_d == 0 && p.hi_d == 127;
        const bool e_ok = span[2] == 0 && relu_e && span[1] - span[0] <= 4 && span[1] <= 24;
        const bool d_ok = span[4] == 0 && relu_d && span[3] - span[5] <= 10;
        if (tid < 4) cst[tid] = tid == 0 ? (e_ok ? span[1] : -1) : (tid == 1 ? (d_ok ? span[3] - 2 : -1) : (tid == 2 ? (p.ce - ch0 > kHalf ? 2 : 1) : span[6]));
        cst[kMultE + tid] = me; cst[kMultD + tid] = md; cst[kUpD + tid] = mine && d_ok ? 1 << (span[3] - sd) : 1;
        cst[kShiftE + tid] = se; cst[kShiftD + tid] = sd;
        cst[kBiasE + tid] = relu_e && !e_ok ? 4 * be : be; cst[kBiasD + tid] = relu_d && !d_ok ? 4 * bd : bd;
        scale_e[tid] = e_ok && mine ? 2 + span[1] - se : 0;
    }
    __syncthreads();
    const bool fast_e = cst[0] >= 0, fast_d = cst[1] >= 0;
    uint32_t invalid = 0;
    // four 2-bit codes at channel k of a packed row, as four int8 of magnitude mag (0 past the row's end)
    auto four = [&](const uint8_t *row, int k, int k_end, uint32_t mag) {
        if (k >= k_end) return 0u;
        const uint32_t b = __ldg(row + (k >> 2));
        invalid |= (b >> 1) & ~b & 0x55u;
        return tc::expand_four(b, mag);
    };
    const int rowb_e = (p.c0 + 3) >> 2, rowb_p = (p.ce + 3) >> 2;
#pragma unroll 4
    for (int i = tid; i < p.ks * kSlice * 8; i += kPrepThreads) {
        const int w = i & 7, n = (i >> 3) & (kSlice - 1), ks = i / (kSlice * 8), ch = ch0 + n;
        const uint32_t v = ch < p.ce ? four(p.we + (size_t)ch * rowb_e, 32 * ks + 4 * w, p.c0, 1u << scale_e[n]) : 0u;
        *reinterpret_cast<uint32_t *>(image + ks * 2 * kTapBytes + tc::swz_offset((uint32_t)n, (uint32_t)w >> 2, 32u) + 4 * (w & 3)) = v;
    }
    for (int i = tid; i < 2 * kSlice * 8; i += kPrepThreads) {
        const int w = i & 7, n = (i >> 3) & (kSlice - 1), d = i / (kSlice * 8);
        const int v = d ? (fast_d ? cst[kBiasD + n] : 0) : (fast_e ? cst[kBiasE + n] << scale_e[n] : 0);
        uint8_t *blk = image + (d ? off_taps(p.ks) + (n / kHalf) * kHalfTaps + 9 * kTapBytes : (uint32_t)p.ks * 2 * kTapBytes);
        *reinterpret_cast<uint32_t *>(blk + tc::swz_offset((uint32_t)(d ? n & (kHalf - 1) : n), (uint32_t)w >> 2, 32u) + 4 * (w & 3)) = tc::bias_word(v, w);
    }
#pragma unroll 4
    for (int i = tid; i < 2 * 9 * kHalf * 2; i += kPrepThreads) {
        const int j = i & 1, n = (i >> 1) & (kHalf - 1), ht = i >> 6, h = ht / 9, tap = ht - 9 * h, ch = ch0 + h * kHalf + n;
        const uint32_t w = ch < p.ce && (n >> 4) == j ? (uint32_t)(uint8_t)__ldg(p.wd + (size_t)ch * 9 + tap) << (8 * (n & 3)) : 0u;
        const int at = (n >> 2) & 3;
        *reinterpret_cast<uint4 *>(image + off_taps(p.ks) + h * kHalfTaps + tap * kTapBytes + tc::swz_offset((uint32_t)n, (uint32_t)j, 32u)) =
            make_uint4(at == 0 ? w : 0u, at == 1 ? w : 0u, at == 2 ? w : 0u, at == 3 ? w : 0u);
    }
#pragma unroll 4
    for (int i = tid; i < p.npad * 16; i += kPrepThreads) {
        const int w = i & 15, o = i >> 4;
        const uint32_t v = o < p.co ? four(p.wp + (size_t)o * rowb_p, ch0 + 4 * w, p.ce, 1u) : 0u;
        *reinterpret_cast<uint32_t *>(image + off_project(p.ks) + tc::swz_offset((uint32_t)o, (uint32_t)w >> 2, 64u) + 4 * (w & 3)) = v;
    }
    for (int i = tid; i < kConstWords; i += kPrepThreads)
        reinterpret_cast<int *>(image + off_consts(p.ks, p.npad))[i] = cst[i];
    if (invalid) raise_status(PROM_ERR_BAD_WEIGHT);
    if (t.behind) ptx::grid_dep_wait();          // complete only once the kernel in front is
}

}}  // namespace prom::block
