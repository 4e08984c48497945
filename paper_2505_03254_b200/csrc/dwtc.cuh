// The int8 depthwise 3x3 convolution (stride 1 and 2) on TMA and the tensor cores.
//
// Channels do not mix in a depthwise convolution, so there is no contraction over channels; the
// contraction is over the nine taps.  A slice is 32 channels; a tile is 128 output columns (16 groups
// of 8 neighbouring pixels of an output row, the groups of all images numbered through), walked down
// the image row by row.  A row of input pixels, stored pixel after pixel with its 32 channels as K, is
// the A operand of an MMA (128 x 32 bytes); shifting it by a tap column dj is nothing but a start
// address, because a group carries its two halo pixels.  B holds three 32 x 32 diagonal blocks, the
// weights w[di][dj] of the three tap rows, so that ONE MMA of shape 128 x 96 x 32 adds an input row's
// contribution to the three output rows that read it, which are neighbours in a ring of accumulator
// blocks (32 columns each) in tensor memory.  An output row so takes four tcgen05.mma.kind::i8: one that
// starts it with the bias (a constant A block against base-127 digits, as in tc.cuh) and three for the
// tap columns.  With stride 2 the even and the odd input columns are two tensor maps, an odd input row
// adds to two output rows (N = 64) and an even one to one (N = 32).
//
// What bounds it: a tap at a time (an MMA of N = 16 or 32 per tap, 9 per output row) is bound by the rate at
// which an SM accepts tcgen05.mma (one per 39 to 54 cycles however small), and 16-byte channel slices
// by the number of L2 requests; with three tap rows per MMA and 64-byte requests the requantiser is
// what is left, and of it what surrounds the arithmetic: read as 32 columns of one row per thread, the
// accumulators met constants in shared memory (two 16-byte loads per four outputs) and left as scattered
// 16-byte pieces.  Measured, us (batch 128; before: a tap at a time, stride 2 on the CUDA cores): 112 x 112 x 32
// 44 -> 31; 56 x 56 x 144 52 -> 37; 56 x 56 x 128 25 (floor at the copy bandwidth 15.7); 28 x 28 x 192 25 -> 13;
// 14 x 14 x 576 21 -> 10; stride 2: 112 x 112 x 96 59 -> 39 (floor 29.4), 28 x 28 x 192 13.3 -> 9.6.  What is left:
// about 5 us of set-up and tail per launch, the rate of 64-byte rows per TMA box (2.2 to 2.8 cycles each), and
// for channel counts that are 16 modulo 32 pixels that straddle 32-byte sectors (144: 37 us against 160: 33).
//
// A CTA (one per SM) owns a block of 64 channels = two slices and a contiguous range of (tile, output
// row).  Warp 0 loads boxes of four input rows, one per group; warps 1 and 2 issue the MMAs of a slice
// each; warps 3..14 are the epilogue: a warp keeps to one quarter of the tile and every third output row;
// four neighbouring threads store the 64 bytes of a pixel.
#pragma once

#include "tc.cuh"

namespace prom { namespace dwtc {

constexpr int kEpiWarps = 12;
constexpr uint32_t kSets = kEpiWarps / 4;        // sets of four warps, one per quarter of a tile
constexpr int kFirstEpi = 3;
constexpr int kThreads = 32 * (kFirstEpi + kEpiWarps);
constexpr int kGroups = 16;                      // groups of 8 output columns in a tile: 128 = one MMA M block
constexpr int kSlice = 32;                       // channels of a slice = K bytes of an MMA
constexpr int kSlices = 2;                       // slices of a CTA's channel block
constexpr int kBlock = kSlice * kSlices;         // 64 channels = bytes of a pixel in shared memory
constexpr int kBoxRows = 4;                      // input rows of a stage
constexpr int kPx = 10;                          // pixels of a group with its halo
constexpr int kRing = 8;                         // accumulator blocks (output rows) per slice
constexpr uint32_t kGroupBytes = kBoxRows * kPx * kBlock;          // 2560: a whole number of swizzle patterns
constexpr uint32_t kEvenBytes = kBoxRows * 8 * kBlock;             // even columns of a group (stride 2)
constexpr uint32_t kTapBytes = 3 * kSlice * kSlice;                // B of one tap column: 96 rows of 32 bytes
constexpr uint32_t kSliceB = 3 * kTapBytes + kSlice * kSlice;      // ... of a slice, with the bias digits

__host__ __device__ constexpr uint32_t stage_bytes(int stride)
{
    return kGroups * (stride == 1 ? kGroupBytes : kGroupBytes + kEvenBytes);
}
__host__ __device__ constexpr int stages(int stride) { return stride == 1 ? 4 : 2; }
__host__ __device__ constexpr uint32_t off_b(int stride) { return (uint32_t)stages(stride) * stage_bytes(stride); }
__host__ __device__ constexpr uint32_t off_aconst(int stride) { return off_b(stride) + kSlices * kSliceB; }
__host__ __device__ constexpr uint32_t off_const(int stride) { return off_aconst(stride) + tc::kAConstBytes; }
__host__ __device__ constexpr uint32_t off_bars(int stride) { return off_const(stride) + kBlock * 16; }
constexpr int kMaxStages = 4;
constexpr int kBars = 2 * kMaxStages + 2 * kRing + 1;
__host__ __device__ constexpr uint32_t smem_bytes(int stride) { return off_bars(stride) + 8 * kBars + 64 + 1024; }

struct Params {
    int batch, h, w, c;     // input
    int ho, wo;             // output
    int segs;               // groups per output row
    int groups;             // batch * segs
    int blocks;             // channel blocks
    long long rows;         // output rows of all tiles
    int per_worker;         // output rows of a CTA
    const int8_t *wt;       // [c][3][3]
    const int32_t *bias, *mult;
    const int8_t *shift;
    int lo, hi;
    int8_t *y;
    int pdl;                // how it is chained to the previous kernel of the stream (tc.cuh: kPdl*)
};

// The part of a CTA's range that lies in one tile.
struct Segment {
    int tile, y0, rows;
};
__device__ __forceinline__ bool next_segment(const Params &p, long long &pos, long long end, Segment &s)
{
    if (pos >= end) return false;
    s.tile = (int)(pos / p.ho);
    s.y0 = (int)(pos - (long long)s.tile * p.ho);
    const long long left = end - pos;
    s.rows = p.ho - s.y0 < left ? p.ho - s.y0 : (int)left;
    pos += s.rows;
    return true;
}
template <int STRIDE>
__device__ __forceinline__ int input_rows(int rows) { return STRIDE == 1 ? rows + 2 : 2 * rows + 1; }

// K-major operand whose rows of 64 bytes are swizzled over 64 bytes; `group` bytes to the next 8 rows.
__device__ __forceinline__ uint64_t desc_pixels(uint32_t addr, uint32_t group)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(group >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// The channel of a slice that accumulator column `col` holds (the order of the rows of B).  A thread of the
// epilogue gets columns 8 j + 2 c + e (j = 0..3, e = 0..1; c = its place in a quad of threads) of a pixel:
// in this order they are eight neighbouring channels, so a thread needs the constants of eight channels
// per slice, which stay in registers, and after one exchange with the thread two places on it has 16
// neighbouring bytes of the pixel (threads 0 and 1 of the first slice, 2 and 3 of the second).
__device__ __forceinline__ int piece_of(int c) { return c == 1 ? 2 : (c == 2 ? 1 : c); }
__device__ __forceinline__ int channel_of(int col) { return 8 * piece_of((col >> 1) & 3) + 2 * (col >> 3) + (col & 1); }

// The 64-bit definition (any clamp, shift and bias) of the eight channels in one thread's half of a
// tmem_ld_16x32 (u: which of its two pixels).  cst: the slice's constants as in the kernel, at the thread's channels.
__device__ __noinline__ uint2 exact_eight(uint32_t taddr, int u, const int *cst, int lo, int hi)
{
    uint32_t v[16];
    ptx::tmem_ld_16x32(taddr, v);
    ptx::tmem_wait_ld();
    int t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t acc = u == 0 ? v[4 * (i >> 1) + (i & 1)] : v[4 * (i >> 1) + 2 + (i & 1)];
        t[i] = requant_exact((int)acc + cst[i], cst[kBlock + i], cst[2 * kBlock + i], lo, hi);
    }
    return make_uint2(ptx::pack_sat_s8(t[1], t[0], ptx::pack_sat_s8(t[3], t[2], 0u)),
                      ptx::pack_sat_s8(t[5], t[4], ptx::pack_sat_s8(t[7], t[6], 0u)));
}

template <int STRIDE>
__global__ void __launch_bounds__(kThreads, 1)
dw3x3_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap emap, const Params p)
{
    constexpr int kStages = stages(STRIDE);
    constexpr uint32_t kStageBytes = stage_bytes(STRIDE);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t smem_base = ptx::smem_u32(smem);
    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;

    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + off_bars(STRIDE));
    const uint32_t bar_full = ptx::smem_u32(bars);
    const uint32_t bar_empty = bar_full + 8 * kMaxStages;
    const uint32_t bar_tfull = bar_empty + 8 * kMaxStages;          // of a ring position, both slices
    const uint32_t bar_tempty = bar_tfull + 8 * kRing;
    const uint32_t bar_drain = bar_tempty + 8 * kRing;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(bars + kBars);
    volatile int *flags = reinterpret_cast<volatile int *>(bars + kBars) + 2;   // [0] abort, [1 + slice] the slice's common shift, or 0: exact epilogue

    const int blk = blockIdx.x % p.blocks, worker = blockIdx.x / p.blocks;
    const int ch0 = blk * kBlock;                                   // the block's first channel
    const int nsl = p.c - ch0 > kSlice ? 2 : 1;                     // slices with channels
    const long long pos0 = (long long)worker * p.per_worker;
    const long long pos1 = pos0 + p.per_worker < p.rows ? pos0 + p.per_worker : p.rows;

    if (p.pdl != tc::kPdlWait) ptx::grid_dep_launch();

    // ---- prologue (nothing here reads the previous kernel's output) -------------------------
    if (warp == 0) {
        if (lane < kStages) {
            ptx::mbar_init(bar_full + 8 * lane, 1);
            ptx::mbar_init(bar_empty + 8 * lane, nsl);
        }
        if (lane < kRing) {
            ptx::mbar_init(bar_tfull + 8 * lane, nsl);
            ptx::mbar_init(bar_tempty + 8 * lane, 4);
        }
        if (lane == 31) {
            ptx::mbar_init(bar_drain, nsl);
            flags[0] = 0;
            ptx::tma_prefetch_desc(&xmap);
            if (STRIDE == 2) ptx::tma_prefetch_desc(&emap);
        }
        ptx::mbar_init_fence();
    }
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32((const void *)tmem_slot), 512u);
    if (p.pdl == tc::kPdlWait) {
        ptx::grid_dep_wait();
        ptx::grid_dep_launch();
    }
    // The loads need the barriers only: warp 0 announces them and goes ahead, the other warps build B.
    int *cst = reinterpret_cast<int *>(smem + off_const(STRIDE));   // bias, mult, shift, scale: kBlock entries each
    if (warp == 0) {
        __syncwarp();
        ptx::named_arrive(1, kThreads);
    } else {
        const int tid = (int)threadIdx.x - 32;
        constexpr int kBuilders = kThreads - 32;
        // constants: thread i < kBlock has channel ch0 + i
        int cb = 0, cmul = 0, csh = 0;
        const bool mine = tid < kBlock && ch0 + tid < p.c;
        if (mine) {
            cb = __ldg(p.bias + ch0 + tid); cmul = __ldg(p.mult + ch0 + tid); csh = __ldg(p.shift + ch0 + tid);
        }
        // B: per slice and tap column 96 rows of 32 bytes; row 32 * k + n has the weight of channel
        // channel_of(n) at that byte and zeros elsewhere.  Tap rows in the order of the output rows they serve:
        // stride 1: di = 2, 1, 0 (output rows r - 1, r, r + 1); stride 2: di = 2, 0 (odd input rows), 1 (even ones)
        for (int i = tid; i < nsl * 3 * 96; i += kBuilders) {
            const int s = i / 288, r = i - s * 288, dj = r / 96, n = r - dj * 96;
            const int k = n >> 5, ch = channel_of(n & 31);
            const int di = STRIDE == 1 ? 2 - k : (k == 0 ? 2 : k - 1);
            const int gch = ch0 + s * kSlice + ch;
            const uint32_t wv = gch < p.c ? (uint32_t)(uint8_t)__ldg(p.wt + (size_t)gch * 9 + di * 3 + dj) : 0u;
            const uint32_t w = wv << (8 * (ch & 3)), at = (uint32_t)ch >> 2;
            uint8_t *b = smem + off_b(STRIDE) + (size_t)s * kSliceB + (size_t)dj * kTapBytes;
            *reinterpret_cast<uint4 *>(b + tc::swz_offset((uint32_t)n, 0u, 32u)) =
                make_uint4(at == 0 ? w : 0u, at == 1 ? w : 0u, at == 2 ? w : 0u, at == 3 ? w : 0u);
            *reinterpret_cast<uint4 *>(b + tc::swz_offset((uint32_t)n, 1u, 32u)) =
                make_uint4(at == 4 ? w : 0u, at == 5 ? w : 0u, at == 6 ? w : 0u, at == 7 ? w : 0u);
        }
        tc::build_aconst(smem + off_aconst(STRIDE), tid, kBuilders);
        // The one-multiply epilogue shifts all channels of a slice by the same amount, the largest shift
        // (at least 2); a channel with a smaller one has its sum scaled up to it first.  It needs the bias
        // within the digits and the scaled sum, |acc| <= 9 * 2^14 plus the bias, within 31 bits.
        if (tid < kBlock) {
            if (mine && !requant_ok(cb, cmul, csh)) { raise_status(PROM_ERR_BAD_REQUANT); cb = 0; cmul = 0; csh = 0; }
            int smax = mine ? max(csh, 2) : 2;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) smax = max(smax, __shfl_xor_sync(0xFFFFFFFFu, smax, d));
            const int up = mine ? smax - csh : 0;
            const bool slow = cb < -tc::kBiasMax || cb > tc::kBiasMax || up > 10 || p.lo != 0 || p.hi != 127;
            const bool any_slow = __any_sync(0xFFFFFFFFu, slow);
            if ((tid & 31) == 0) flags[1 + tid / kSlice] = any_slow ? 0 : smax;
            cst[tid] = cb; cst[kBlock + tid] = cmul; cst[2 * kBlock + tid] = csh; cst[3 * kBlock + tid] = 1 << (up & 31);
        }
        ptx::named_sync(2, kBuilders);
        // bias digits: a row per column, 32 digits of which the first has weight 1 (the second stays 0), the
        // others 127; a thread writes four
        const bool in_sum = flags[1] != 0 && (nsl == 1 || flags[2] != 0);     // both slices or neither
        for (int i = tid; i < kBlock * 8; i += kBuilders) {
            const int col = i >> 3, w = i & 7, s = col / kSlice;
            const int b = in_sum ? cst[s * kSlice + channel_of(col & 31)] : 0;
            uint8_t *bb = smem + off_b(STRIDE) + (size_t)s * kSliceB + 3 * kTapBytes;
            *reinterpret_cast<uint32_t *>(bb + tc::swz_offset((uint32_t)(col & 31), (uint32_t)w >> 2, 32u) + 4 * (w & 3)) = tc::bias_word(b, w);
        }
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before_sync();
        ptx::named_sync(1, kThreads);
        ptx::tc_fence_after_sync();
    }
    const uint32_t tmem_base = warp == 0 ? 0u : *tmem_slot;

    if (warp == 0) {
        // ---- TMA producer: lane g loads the boxes of group g ----------------------------------
        uint32_t slot = 0, ph = 0, issued = 0;
        bool ok = true;
        if (p.pdl == tc::kPdlChain) ptx::grid_dep_wait();      // the loads are the only reads of x
        long long pos = pos0;
        Segment sg;
        while (ok && next_segment(p, pos, pos1, sg)) {
            const int g = sg.tile * kGroups + (lane & 15);
            const int img = g / p.segs, seg = g - img * p.segs;    // a group past the last is past the last image
            const int nin = input_rows<STRIDE>(sg.rows);
            int y = sg.y0 * STRIDE - 1;
            for (int j = 0; j < nin; j += kBoxRows, y += kBoxRows) {
                if (!tc::wait_bar_warp(bar_empty + 8 * slot, ph ^ 1u, flags)) { ok = false; break; }
                const uint32_t bfull = bar_full + 8 * slot, dst = smem_base + slot * kStageBytes;
                if (lane == 0) ptx::mbar_expect_tx(bfull, kStageBytes);
                __syncwarp();
                if (lane < kGroups) {
                    // {channel, column, row, image}; the halo starts one pixel to the left
                    ptx::tma_load_4d(dst + lane * kGroupBytes, &xmap, ch0, seg * 8 - 1, y, img, bfull);
                    if (STRIDE == 2)
                        ptx::tma_load_4d(dst + kGroups * kGroupBytes + lane * kEvenBytes, &emap, ch0, seg * 8, y, img, bfull);
                }
                ++issued;
                if (++slot == kStages) { slot = 0; ph ^= 1u; }
            }
        }
        if (lane == 0) tc::drain_copies(bar_full, kStages, issued);
        __syncwarp();
    } else if (warp < kFirstEpi) {
        // ---- MMA issuers: warp 1 slice 0, warp 2 slice 1 ----------------------------------------
        const int s = warp - 1;
        if (s < nsl) {                                    // the whole warp; one lane issues
            const bool leader = ptx::elect_one();
            // s8 x s8 -> s32, both K-major, M = 128; N in blocks of 32
            constexpr uint32_t kI0 = (2u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
            constexpr uint32_t kN32 = (uint32_t)(kSlice >> 3) << 17;
            const uint64_t d32 = tc::smem_desc(0u, 32u);
            const uint64_t ac = d32 | (uint64_t)((smem_base + off_aconst(STRIDE)) >> 4);
            const uint32_t b0 = (smem_base + off_b(STRIDE) + (uint32_t)s * kSliceB) >> 4;
            const uint64_t wb = d32 | (uint64_t)(b0 + ((3 * kTapBytes) >> 4));
            const uint32_t acc0 = tmem_base + (uint32_t)s * kRing * kSlice;
            const uint32_t tf = bar_tfull, te = bar_tempty;
            uint32_t slot = 0, ph = 0;
            uint32_t rp = 0, rph = 1;       // ring position of the next output row, parity of its empty barrier
            bool ok = true;

            // The three tap columns of one input row: `cnt` output rows whose accumulators are neighbours in
            // the ring from position r0 on (in two pieces where they wrap), B from tap-row block bk on.
            auto taps = [&](uint32_t a_px, uint32_t a_even, uint32_t r0, uint32_t cnt, uint32_t bk) {
                const uint32_t bb = b0 + ((bk * kSlice * kSlice) >> 4);
                const uint32_t cnt1 = r0 + cnt > kRing ? kRing - r0 : cnt;
                const uint32_t d = acc0 + r0 * kSlice, i1 = kI0 | (cnt1 * kN32);
#pragma unroll
                for (uint32_t dj = 0; dj < 3; ++dj) {
                    uint64_t a;
                    if (STRIDE == 1) a = desc_pixels(a_px + dj * kBlock, kGroupBytes);
                    else if (dj == 1) a = desc_pixels(a_even, kEvenBytes);
                    else a = desc_pixels(a_px + (dj >> 1) * kBlock, kGroupBytes);
                    const uint32_t b = bb + ((dj * kTapBytes) >> 4);
                    if (leader) ptx::mma_i8<true>(d, a, d32 | (uint64_t)b, i1);
                    if (cnt1 < cnt && leader)
                        ptx::mma_i8<true>(acc0, a, d32 | (uint64_t)(b + ((cnt1 * kSlice * kSlice) >> 4)), kI0 | ((cnt - cnt1) * kN32));
                }
            };
            // Begins the output row at ring position rp: waits until its accumulator is free, then the bias.
            auto begin_row = [&] {
                if (!tc::wait_bar_warp(te + 8 * rp, rph, flags)) return false;
                ptx::tc_fence_after_sync();
                if (leader) ptx::mma_i8<false>(acc0 + rp * kSlice, ac, wb, kI0 | kN32);
                return true;
            };

            long long pos = pos0;
            Segment sg;
            while (ok && next_segment(p, pos, pos1, sg)) {
                const int nin = input_rows<STRIDE>(sg.rows), last = sg.rows - 1;
                for (int j0 = 0; j0 < nin && ok; j0 += kBoxRows) {
                    if (!tc::wait_bar_warp(bar_full + 8 * slot, ph, flags)) { ok = false; break; }
                    ptx::tc_fence_after_sync();
                    const uint32_t stage = smem_base + slot * kStageBytes + (uint32_t)s * kSlice;
#pragma unroll
                    for (int jr = 0; jr < kBoxRows; ++jr) {
                        const int j = j0 + jr;
                        if (j >= nin) break;
                        const uint32_t a_px = stage + (uint32_t)jr * (kPx * kBlock);
                        const uint32_t a_even = stage + kGroups * kGroupBytes + (uint32_t)jr * (8 * kBlock);
                        if (STRIDE == 1) {
                            // input row j - 1 of the segment: output rows j - 2, j - 1 and j, which it begins
                            const bool fresh = j <= last;
                            if (fresh && !begin_row()) { ok = false; break; }
                            if (j >= 2 && fresh) {
                                taps(a_px, 0u, (rp - 2) & (kRing - 1), 3, 0);
                            } else {
                                const int lo = j >= 2 ? j - 2 : 0, hi = fresh ? j : last;
                                taps(a_px, 0u, (rp - (uint32_t)(fresh ? j - lo : last + 1 - lo)) & (kRing - 1), (uint32_t)(hi - lo + 1), (uint32_t)(2 - (j - lo)));
                            }
                            if (j >= 2 && leader) ptx::mma_commit(tf + 8 * ((rp - (fresh ? 2u : (uint32_t)(last + 1 - (j - 2)))) & (kRing - 1)));
                            if (fresh && ++rp == kRing) { rp = 0; rph ^= 1u; }
                        } else if (jr & 1) {
                            // even input row: the newest output row alone, which the odd row before it began
                            taps(a_px, a_even, (rp - 1) & (kRing - 1), 1, 2);
                        } else {
                            // odd input row: finishes output row j / 2 - 1 and begins j / 2
                            const bool fresh = (j >> 1) <= last, old = j > 0;
                            if (fresh && !begin_row()) { ok = false; break; }
                            taps(a_px, a_even, (rp - (old ? 1u : 0u)) & (kRing - 1), (old ? 1u : 0u) + (fresh ? 1u : 0u), old ? 0u : 1u);
                            if (old && leader) ptx::mma_commit(tf + 8 * ((rp - 1) & (kRing - 1)));
                            if (fresh && ++rp == kRing) { rp = 0; rph ^= 1u; }
                        }
                    }
                    if (leader) ptx::mma_commit(bar_empty + 8 * slot);
                    if (++slot == kStages) { slot = 0; ph ^= 1u; }
                }
            }
            // every MMA has finished before tensor memory is released
            if (leader) ptx::mma_commit(bar_drain);
            const unsigned long long g0 = ptx::globaltimer();
            while (!ptx::mbar_try_wait(bar_drain, 0) && ptx::globaltimer() - g0 < tc::kWaitLimitNs) {}
        }
        __syncwarp();
    } else {
        // ---- epilogue -----------------------------------------------------------------------------
        // Sets of four warps (one per quarter of the tile) take the output rows in turn.
        const int q = warp & 3;
        const uint32_t first = (uint32_t)(warp - kFirstEpi) >> 2;
        const int c = lane & 3, px = lane >> 2;         // this thread's place in its quad, its pixel of every group
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        const bool some = ch0 + c * 16 < p.c && c < 2 * nsl;      // whether there are channels at its 16 bytes
        const int down0 = flags[1] - 2, down1 = flags[2] - 2;     // negative: exact epilogue
        const bool fast = down0 >= 0 && (nsl == 1 || down1 >= 0);
        const int *cmy = cst + 8 * piece_of(c);         // this thread's channels of the first slice
        int mu0[8], up0[8], mu1[8], up1[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            mu0[i] = cmy[kBlock + i]; up0[i] = cmy[3 * kBlock + i];
            mu1[i] = cmy[kBlock + kSlice + i]; up1[i] = cmy[3 * kBlock + kSlice + i];
        }
        const size_t pitch = (size_t)p.wo * p.c;

        // Eight channels of one pixel, clamp [0, 127], bias already in the sum.  The sum scaled to the slice's
        // common shift, one high word of a 64-bit multiply-add (rounding term in the addend), one shift:
        // floor(p / 2^(30 + shift)) + 1, twice the rounded value, kept through a saturating pack to [0, 255] and halved.
        auto eight = [&](const uint32_t (&v)[16], int u, const int (&mu)[8], const int (&up)[8], int down) {
            const long long r64 = (long long)(1u << down) << 32;
            int t[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                t[i] = (int)(((long long)((int)v[4 * (i >> 1) + 2 * u + (i & 1)] * up[i]) * mu[i] + r64) >> 32) >> down;
            return make_uint2((ptx::pack_sat_u8(t[1], t[0], ptx::pack_sat_u8(t[3], t[2], 0u)) >> 1) & 0x7F7F7F7Fu,
                              (ptx::pack_sat_u8(t[5], t[4], ptx::pack_sat_u8(t[7], t[6], 0u)) >> 1) & 0x7F7F7F7Fu);
        };
        // The pixel's bytes of both slices in the quad: every thread keeps eight, gets eight and stores 16.
        auto store = [&](uint2 a, uint2 b, int8_t *y) {
            const uint2 give = c < 2 ? b : a, keep = c < 2 ? a : b;
            const uint2 got = make_uint2(__shfl_xor_sync(0xFFFFFFFFu, give.x, 2), __shfl_xor_sync(0xFFFFFFFFu, give.y, 2));
            if (y)
                *reinterpret_cast<uint4 *>(y) = c < 2 ? make_uint4(keep.x, keep.y, got.x, got.y)
                                                      : make_uint4(got.x, got.y, keep.x, keep.y);
        };

        bool ok = true;
        uint32_t k = 0;                                 // output rows of the segments before
        long long pos = pos0;
        Segment sg;
        while (ok && next_segment(p, pos, pos1, sg)) {
            // this thread's pixel of each of the warp's four groups (null: outside the image)
            int8_t *yg[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int g = sg.tile * kGroups + q * 4 + i;
                const int img = g / p.segs, ox = (g - img * p.segs) * 8 + px;
                yg[i] = some && g < p.groups && ox < p.wo
                            ? p.y + (((size_t)img * p.ho + sg.y0) * p.wo + ox) * (size_t)p.c + ch0 + 16 * c
                            : nullptr;
            }
            const uint32_t kseg = k;
            k += (uint32_t)sg.rows;
            for (uint32_t kk = kseg + (first + kSets - kseg % kSets) % kSets; kk < k; kk += kSets) {
                const uint32_t r = kk & (kRing - 1), acc0 = t_lane + r * kSlice, acc1 = acc0 + kRing * kSlice;
                const size_t off = (size_t)(kk - kseg) * pitch;
                ok = __all_sync(0xFFFFFFFFu, tc::wait_bar<true>(bar_tfull + 8 * r, (kk / kRing) & 1u, flags));
                if (!ok) break;
                ptx::tc_fence_after_sync();
                auto at = [&](int i) { return yg[i] ? yg[i] + off : nullptr; };
                if (!fast) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t half = (uint32_t)(i >> 1) << 20;          // the upper 16 lanes
                        const uint2 a = exact_eight(acc0 + half, i & 1, cmy, p.lo, p.hi);
                        const uint2 b = nsl == 2 ? exact_eight(acc1 + half, i & 1, cmy + kSlice, p.lo, p.hi) : a;
                        store(a, b, at(i));
                    }
                    tc::release_acc(bar_tempty + 8 * r);
                    continue;
                }
                // accumulators of the next pieces are on their way while a piece is worked on
                uint32_t va[16], vb[16];
                ptx::tmem_ld_16x32(acc0, va);
                if (nsl == 2) ptx::tmem_ld_16x32(acc1, vb);
                ptx::tmem_wait_ld();
                uint2 a0 = eight(va, 0, mu0, up0, down0), a1 = eight(va, 1, mu0, up0, down0);
                ptx::tmem_ld_16x32(acc0 + (16u << 16), va);
                uint2 b0 = a0, b1 = a1;
                if (nsl == 2) { b0 = eight(vb, 0, mu1, up1, down1); b1 = eight(vb, 1, mu1, up1, down1); }
                if (nsl == 2) ptx::tmem_ld_16x32(acc1 + (16u << 16), vb);
                store(a0, b0, at(0));
                store(a1, b1, at(1));
                ptx::tmem_wait_ld();
                tc::release_acc(bar_tempty + 8 * r);
                b0 = a0 = eight(va, 0, mu0, up0, down0);
                b1 = a1 = eight(va, 1, mu0, up0, down0);
                if (nsl == 2) { b0 = eight(vb, 0, mu1, up1, down1); b1 = eight(vb, 1, mu1, up1, down1); }
                store(a0, b0, at(2));
                store(a1, b1, at(3));
            }
        }
    }

    // ---- teardown -------------------------------------------------------------------------------
    // every CTA waits for the previous kernel before it ends, also one whose loader had no row
    if (p.pdl == tc::kPdlChain && threadIdx.x == 32) ptx::grid_dep_wait();
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, 512u);
    }
}

}}  // namespace prom::dwtc
