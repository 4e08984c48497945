// The tensor-core variant for layers whose contraction, not their bytes, is the bound
// (many input and many output channels on many rows).
//
// tc_conv_kernel keeps the weights of a channel group resident and streams the activations
// past them once per group; with Cin x Cout in the hundreds of thousands a group is only a few
// dozen channels wide, the MMAs are narrow and the activations cross the SM many times.  Here
// the roles are swapped: a pair of CTAs (one per SM) keeps a tile of 256 rows resident, all of its K
// (up to 8 chunks of 128 bytes, 128 rows in each CTA), and streams the expanded weights of one
// 256-channel column tile after the other through a ring.  The MMAs span the pair (cta_group::2,
// 256 x 256 x 32): each CTA holds half of a column tile's weights, so that per 128 clocks of the tensor
// pipe a CTA's shared memory is read for 4 KB of rows and 4 KB of weights and written with 4 KB, 96 of the
// 128 bytes per clock that it can take, and 32 bytes per clock come from L2.  (One CTA alone with 128 x 128 x 32
// MMAs needs 128 + 64 bytes per clock, and 64 from L2, of which 58 to 61 were measured.)
// 1.6 M x 960 -> 1280: 1615-1670 us with single CTAs, 1460-1480 with pairs, under the power cap in both.
//
// wide_prep_kernel (kPrepParts CTAs per 128 channels) expands the 2-bit weights into an int8 matrix
// [Cout padded to 128][Cin padded to 128] in global scratch, scaled for the one-multiply
// epilogue of tc.cuh where the tile's constants allow it, and writes the tile's bias digits
// and requantisation constants beside it.  The convolution kernel reads that matrix through a
// tensor map (128-byte swizzle, like the activations), the bias digits as the last "chunk" of a
// column tile, and the constants into a small ring of their own.
//
// Warp 0 of each CTA loads its weights, warp 18 its rows and constants, each waiting only for room of its own (one
// loader for all three held the weights back until the constants of the unit before last had been read, which put
// half of every read-out on the MMAs' path).  The chunks of rows go through a ring of eight, so that with K of less
// than eight chunks the next tile's first ones are there before this tile's last unit has ended.
// Warp 1 of the first CTA issues the MMAs of both, warps 2..17 requantise the
// CTA's own 128 rows, 32 columns at a time, and store through the output's tensor map (rows and columns outside
// the matrix are not written).
#pragma once

#include "tc.cuh"

namespace prom { namespace wide {

constexpr int kEpiWarps = 16;                     // four groups of four
constexpr int kLoader2 = 2 + kEpiWarps;           // warp of the second loader
constexpr int kThreads = 32 * (kLoader2 + 1);     // weight loader, MMA issuer, epilogue warps, loader of rows and constants
constexpr int kNt = 128;                          // channels of a block of constants
constexpr int kChunk = 128;                       // bytes of K per chunk = swizzle span
constexpr int kMaxKc = 8;                         // resident K chunks: Cin <= 1024
constexpr int kASlots = kMaxKc;                   // their ring (a power of two)
constexpr int kMaxStages = 8;
constexpr int kAccs = 2;                          // accumulators of up to 256 columns
constexpr uint32_t kAChunkBytes = 128 * kChunk;   // one resident chunk of a CTA's 128 rows
constexpr uint32_t kWbiasBytes = kNt * 32;        // bias digits of a block (32-byte swizzled rows)
// constants of a block: mult[128], {bias, shift}[128], header {shmax, fast, bad, clamp}
constexpr uint32_t kConstBytes = kNt * 4 + kNt * 8 + 16 + 112;
constexpr uint32_t kEpiCols = 32;                 // columns an epilogue warp stages per store
constexpr uint32_t kSlabBytes = 32 * kEpiCols;
constexpr int kBars = 2 * kASlots + 2 * kMaxStages + 4 * kAccs + 1;

struct Params {
    long long m;
    int cin, cout;
    int kc, ksteps_last;        // chunks of K; 32-byte MMA steps in the last one
    int n_mtiles, n_ctiles;     // tiles of 256 rows, column tiles
    int nb;                     // 128-channel blocks per column tile: 1 or 2
    int stages;                 // of the weight ring
    uint32_t off_w, off_const, off_out, off_aconst, off_bars;
    const uint8_t *consts;      // [n_ctiles * nb][kConstBytes]
    int act_min, act_max;
};

struct PrepParams {
    int cin, cout, k_pad;
    const uint8_t *w_packed;
    const int32_t *bias, *mult;
    const int8_t *shift;
    int act_min, act_max;
    int signed_fast;            // the reader of the constants has the one-multiply form for [-128, 127] too
    int8_t *w8;                 // [n_ctiles * 128][k_pad]
    uint8_t *wbias, *consts;
};

// Operands are for one clamp; the kernel that reads them is told it again.
__device__ __forceinline__ int clamp_code(int lo, int hi) { return ((lo & 0xFF) << 8) | (hi & 0xFF); }

// The operands of column tile `tile` of one layer; all 256 threads of the CTA take part.  `parts` CTAs share
// the expansion of the tile's weights (each checks the constants; the first writes them).
__device__ __forceinline__ void prep_tile(const PrepParams &p, const int tile, const int part = 0, const int parts = 1)
{
    __shared__ int s_mult[kNt], s_bias[kNt], s_shift[kNt];
    __shared__ int s_flags[4];      // shmin, shmax, bad, slow
    const int n0 = tile * kNt;
    if (threadIdx.x == 0) { s_flags[0] = 31; s_flags[1] = 0; s_flags[2] = 0; s_flags[3] = 0; }
    __syncthreads();
    if (threadIdx.x < kNt) {
        const int n = n0 + threadIdx.x;
        int b = 0, mu = 0, sh = 0;
        if (n < p.cout) {
            b = __ldg(p.bias + n); mu = __ldg(p.mult + n); sh = __ldg(p.shift + n);
            if (!requant_ok(b, mu, sh)) { s_flags[2] = 1; b = 0; mu = 0; sh = 0; }
            atomicMin(&s_flags[0], sh);
            atomicMax(&s_flags[1], sh);
            // the one-multiply epilogue needs |acc + bias| * 2^6 below 2^31 and the scaled bias
            // within the range of its digits
            const long long ab = b < 0 ? -(long long)b : b;
            if ((((long long)128 * p.cin + ab) << 6) >= (1ll << 31) || (ab << 6) > tc::kBiasMax) s_flags[3] = 1;
        }
        s_mult[threadIdx.x] = mu; s_bias[threadIdx.x] = b; s_shift[threadIdx.x] = sh;
    }
    __syncthreads();
    const int shmax = s_flags[1];
    const bool bad = s_flags[2] != 0;
    const bool fast = !bad && s_flags[3] == 0 && (p.act_min == 0 || (p.signed_fast && p.act_min == -128)) && p.act_max == 127 && shmax - s_flags[0] <= 4 &&
                      shmax <= 24 && s_flags[0] <= shmax;
    if (bad && threadIdx.x == 0) raise_status(PROM_ERR_BAD_REQUANT);

    // constants and bias digits
    uint8_t *cst = p.consts + (size_t)tile * kConstBytes;
    uint8_t *wb = p.wbias + (size_t)tile * kWbiasBytes;
    if (threadIdx.x < kNt && part == 0) {
        const int c = threadIdx.x;
        reinterpret_cast<int *>(cst)[c] = s_mult[c];
        reinterpret_cast<int2 *>(cst + kNt * 4)[c] = make_int2(s_bias[c], s_shift[c]);
        uint32_t wd[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (fast && n0 + c < p.cout) {
            const int v = s_bias[c] << (2 + shmax - s_shift[c]);
            int h = (v >= 0 ? v + 63 : v - 63) / 127;        // nearest multiple of 127
            const int lo = v - 127 * h;                       // within [-63, 63]
            wd[0] = (uint32_t)lo & 0xFFu;
            for (int d = 0; d < tc::kBiasHiDigits; ++d) {
                const int dig = h > 127 ? 127 : (h < -127 ? -127 : h);
                h -= dig;
                const int k = d + 2;
                wd[k >> 2] |= ((uint32_t)dig & 0xFFu) << (8 * (k & 3));
            }
        }
        *reinterpret_cast<uint4 *>(wb + tc::swz_offset((uint32_t)c, 0u, 32u)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
        *reinterpret_cast<uint4 *>(wb + tc::swz_offset((uint32_t)c, 1u, 32u)) = make_uint4(wd[4], wd[5], wd[6], wd[7]);
    }
    if (threadIdx.x == 0 && part == 0) {
        int *hdr = reinterpret_cast<int *>(cst + kNt * 12);
        hdr[0] = shmax; hdr[1] = fast ? 1 : 0; hdr[2] = bad ? 1 : 0; hdr[3] = clamp_code(p.act_min, p.act_max);
    }

    // the tile's rows of the int8 matrix, 16 bytes (16 codes = one 32-bit word) per step
    const int rowb = (p.cin + 3) >> 2, pieces = p.k_pad >> 4;
    uint32_t invalid = 0;
    for (int i = part * blockDim.x + threadIdx.x; i < kNt * pieces; i += parts * blockDim.x) {
        const int c = i / pieces, j = i - c * pieces, n = n0 + c;
        uint4 val = make_uint4(0u, 0u, 0u, 0u);
        if (n < p.cout && j * 16 < p.cin && !bad) {
            const uint32_t w = *reinterpret_cast<const uint32_t *>(p.w_packed + (size_t)n * rowb + j * 4);
            invalid |= (w >> 1) & ~w & 0x55555555u;
            const uint32_t mag = fast ? (4u << (shmax - s_shift[c])) : 1u, neg = 256u - mag;
            uint32_t wd[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const uint32_t code = (w >> (2 * e)) & 3u;
                const uint32_t byte = code == 1u ? mag : (code == 3u ? neg : 0u);
                wd[e >> 2] |= byte << (8 * (e & 3));
            }
            val = make_uint4(wd[0], wd[1], wd[2], wd[3]);
        }
        *reinterpret_cast<uint4 *>(p.w8 + (size_t)n * p.k_pad + j * 16) = val;
    }
    if (invalid) raise_status(PROM_ERR_BAD_WEIGHT);
}

// kPrepParts CTAs per column tile (one per tile kept 138 SMs idle for 15 us).
constexpr int kPrepParts = 8;
__global__ void __launch_bounds__(256, 1) wide_prep_kernel(const PrepParams p)
{
    // launched with programmatic dependent launch: the weights may be the previous kernel's output, and the
    // scratch it fills may still be read by an earlier call
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    prep_tile(p, (int)blockIdx.x / kPrepParts, (int)blockIdx.x % kPrepParts, kPrepParts);
}

// The same for several layers in one launch: CTA b belongs to the layer l with first[l] <= b < first[l + 1].
constexpr int kMaxPrepLayers = 16;
struct PrepBatch {
    int n;
    int first[kMaxPrepLayers + 1];
    PrepParams layer[kMaxPrepLayers];
};

__global__ void __launch_bounds__(256, 1) wide_prep_batch_kernel(const __grid_constant__ PrepBatch t)
{
    int l = 0;
    while (l + 1 < t.n && (int)blockIdx.x >= t.first[l + 1]) ++l;
    prep_tile(t.layer[l], (int)blockIdx.x - t.first[l]);
}

// A loader that has given up must not let its CTA go while its copies are in flight.  They are counted on barriers of the
// first CTA, together with the other CTA's, which may never be issued, so there is no phase to wait for: it waits for
// as long as tc::drain_copies would at most.
__device__ __noinline__ void outwait_copies()
{
    const unsigned long long t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < tc::kWaitLimitNs) {}
}

// One pair of CTAs per two SMs takes a contiguous range of units (row tile of 256, column tile), column tiles
// of a row tile one after the other; the range's first unit in a row tile loads the tile's rows, the last one
// lets go of them.  (Ranges instead of whole row tiles: 98 row tiles on 74 pairs are 1.3 rounds instead of 2.)
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
wide_conv_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap,
                 const __grid_constant__ CUtensorMap bmap, const __grid_constant__ CUtensorMap ymap, const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t smem_base = ptx::smem_u32(smem);
    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_rank();

    // Barriers of the first CTA count both CTAs' loads (afull, wfull) and read-outs (tempty); the MMAs'
    // completions arrive in both (aempty, wempty, tfull); constants are each CTA's own.
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + p.off_bars);
    const uint32_t bar_afull = ptx::smem_u32(bars);               // a resident chunk has landed
    const uint32_t bar_aempty = bar_afull + 8 * kASlots;           // ... has been read for the last time
    const uint32_t bar_wfull = bar_aempty + 8 * kASlots;           // weight ring
    const uint32_t bar_wempty = bar_wfull + 8 * kMaxStages;
    const uint32_t bar_tfull = bar_wempty + 8 * kMaxStages;       // accumulators
    const uint32_t bar_tempty = bar_tfull + 8 * kAccs;
    const uint32_t bar_cfull = bar_tempty + 8 * kAccs;            // constants of a unit (slot = accumulator)
    const uint32_t bar_cempty = bar_cfull + 8 * kAccs;
    const uint32_t bar_drain = bar_cempty + 8 * kAccs;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(bars + kBars);
    volatile int *flags = reinterpret_cast<volatile int *>(bars + kBars + 1);     // [0] abort

    const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
    const long long units = (long long)p.n_mtiles * p.n_ctiles;
    const long long u0 = units * pair / pairs, u1 = units * (pair + 1) / pairs;
    const int mt0 = (int)(u0 / p.n_ctiles), ct0 = (int)(u0 % p.n_ctiles), n_units = (int)(u1 - u0);
    const int nt = p.nb * kNt;
    const uint32_t w_stage = (uint32_t)(nt / 2) * kChunk;
    // columns of column tile ct that exist, in the MMA's steps of 32
    auto width = [&](int ct) { const int left = p.cout - ct * nt; return left >= nt ? nt : (left + 31) & ~31; };

    // ---- prologue -----------------------------------------------------------------------------
    if (warp == 0) {
        if (lane < kASlots) {
            ptx::mbar_init(bar_afull + 8 * lane, 1);
            ptx::mbar_init(bar_aempty + 8 * lane, 1);
        } else if (lane < kASlots + kMaxStages) {
            ptx::mbar_init(bar_wfull + 8 * (lane - kASlots), 1);
            ptx::mbar_init(bar_wempty + 8 * (lane - kASlots), 1);
        } else if (lane < kASlots + kMaxStages + kAccs) {
            const int b = lane - kASlots - kMaxStages;
            ptx::mbar_init(bar_tfull + 8 * b, 1);
            ptx::mbar_init(bar_tempty + 8 * b, 2 * kEpiWarps);
            ptx::mbar_init(bar_cfull + 8 * b, 1);
            ptx::mbar_init(bar_cempty + 8 * b, kEpiWarps);
        } else if (lane == 31) {
            ptx::mbar_init(bar_drain, 1);
            flags[0] = 0;
            ptx::tma_prefetch_desc(&xmap);
            ptx::tma_prefetch_desc(&wmap);
            ptx::tma_prefetch_desc(&bmap);
            ptx::tma_prefetch_desc(&ymap);
        }
        ptx::mbar_init_fence();
    }
    if (warp == 1) ptx::tmem_alloc_pair(ptx::smem_u32((const void *)tmem_slot), 512u);
    tc::build_aconst(smem + p.off_aconst, (int)threadIdx.x, kThreads);
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // The next call's kernel may start its set-up; it waits before it reads or writes anything.  (Not before the
    // tensor memory is held, which that kernel may want too.)
    ptx::grid_dep_launch();

    if (warp == 0) {
        // ---- loader of weights ----------------------------------------------------------------------
        // Per unit this CTA's half of the column tile's weights, chunk by chunk, then of the bias digits.
        {
            const bool leader = ptx::elect_one();
            ptx::grid_dep_wait();           // for wide_prep_kernel, which waited for what wrote x
            const uint32_t wfull = ptx::map_to_rank(bar_wfull, 0);
            uint32_t st = 0, ph = 0;
            int ct = ct0;
            bool ok = true;
            // the ring's next stage, armed for both CTAs' loads
            auto next_stage = [&](uint32_t tx, uint32_t &bar) -> uint32_t {
                if (!tc::wait_bar_warp(bar_wempty + 8 * st, ph ^ 1u, flags)) { ok = false; return 0u; }
                if (leader && rank == 0) ptx::mbar_expect_tx(bar_wfull + 8 * st, 2u * tx);
                bar = wfull + 8 * st;
                const uint32_t dst = smem_base + p.off_w + st * w_stage;
                if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
                return dst;
            };
            for (int k = 0; k < n_units && ok; ++k) {
                const int w_row = ct * nt + (int)rank * (width(ct) / 2);
                for (int c = 0; c < p.kc && ok; ++c) {
                    uint32_t bar = 0;
                    const uint32_t dst = next_stage(w_stage, bar);
                    if (ok && leader) ptx::tma_load_2d_pair(dst, &wmap, c * kChunk, w_row, bar);
                }
                if (ok) {
                    uint32_t bar = 0;
                    const uint32_t dst = next_stage((uint32_t)(nt / 2) * 32u, bar);
                    if (ok && leader) ptx::tma_load_2d_pair(dst, &bmap, 0, w_row, bar);
                }
                if (++ct == p.n_ctiles) ct = 0;
            }
            // The completions of the last MMAs must have arrived here before the CTA may go away.
            for (int s = 0; s < p.stages && ok; ++s) {
                ok = tc::wait_bar_warp(bar_wempty + 8 * st, ph ^ 1u, flags);
                if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
            }
            if (!ok) outwait_copies();
        }
        __syncwarp();
    } else if (warp == kLoader2) {
        // ---- loader of rows and constants -------------------------------------------------------------
        // Per unit: this CTA's rows, for the first unit of a row tile, then the constants.
        {
            const bool leader = ptx::elect_one();
            ptx::grid_dep_wait();
            const uint32_t afull = ptx::map_to_rank(bar_afull, 0);
            uint32_t n = 0;                 // chunks of rows so far
            int mt = mt0, ct = ct0;
            bool ok = true;
            for (int k = 0; k < n_units && ok; ++k) {
                if (k == 0 || ct == 0) {
                    for (int c = 0; c < p.kc; ++c, ++n) {
                        const uint32_t s = n % kASlots;
                        if (!tc::wait_bar_warp(bar_aempty + 8 * s, ((n / kASlots) & 1u) ^ 1u, flags)) { ok = false; break; }
                        if (leader) {
                            if (rank == 0) ptx::mbar_expect_tx(bar_afull + 8 * s, 2u * kAChunkBytes);
                            ptx::tma_load_2d_pair(smem_base + s * kAChunkBytes, &xmap, c * kChunk, mt * 256 + (int)rank * 128, afull + 8 * s);
                        }
                    }
                    if (!ok) break;
                }
                const uint32_t slot = (uint32_t)k & 1u;
                if (!tc::wait_bar_warp(bar_cempty + 8 * slot, (((uint32_t)k >> 1) & 1u) ^ 1u, flags)) { ok = false; break; }
                if (leader) {
                    const uint32_t bytes = (uint32_t)p.nb * kConstBytes;
                    ptx::mbar_expect_tx(bar_cfull + 8 * slot, bytes);
                    ptx::bulk_load(smem_base + p.off_const + slot * bytes, p.consts + (size_t)ct * bytes, bytes, bar_cfull + 8 * slot);
                }
                if (++ct == p.n_ctiles) { ct = 0; ++mt; }
            }
            for (int s = 0; s < kASlots && ok; ++s, ++n)
                ok = tc::wait_bar_warp(bar_aempty + 8 * (n % kASlots), ((n / kASlots) & 1u) ^ 1u, flags);
            if (!ok) outwait_copies();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer: the first CTA's, for both --------------------------------------------------
        // (the whole warp, one lane issues: descriptors then stay in uniform registers)
        if (rank == 0) {
            const bool leader = ptx::elect_one();
            const uint64_t d_128 = tc::smem_desc(0u, 128u), d_32 = tc::smem_desc(0u, 32u);
            const uint64_t ac_desc = d_32 | (uint64_t)((smem_base + p.off_aconst) >> 4);
            const uint32_t a_lo0 = smem_base >> 4, w_lo0 = (smem_base + p.off_w) >> 4;
            const uint32_t a_step = kAChunkBytes >> 4, w_step = w_stage >> 4;
            uint32_t st = 0, ph = 0, n0 = 0;          // n0: chunks of rows before this row tile's
            int ct = ct0, k = 0;
            bool ok = true;
            for (; k < n_units && ok; ++k) {
                const uint32_t acc = (uint32_t)k & 1u;
                // s8 x s8 -> s32, both K-major, M = 256
                const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | (((uint32_t)width(ct) >> 3) << 17) | ((256u >> 4) << 24);
                if (!tc::wait_bar_warp(bar_tempty + 8 * acc, (((uint32_t)k >> 1) & 1u) ^ 1u, flags)) { ok = false; break; }
                ptx::tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * 256u;
                const bool first = k == 0 || ct == 0, last = k + 1 == n_units || ct + 1 == p.n_ctiles;     // of the row tile
                for (int c = 0; c < p.kc; ++c) {
                    const uint32_t s = (n0 + (uint32_t)c) % kASlots;
                    if (first && !tc::wait_bar_warp(bar_afull + 8 * s, ((n0 + (uint32_t)c) / kASlots) & 1u, flags)) { ok = false; break; }
                    if (!tc::wait_bar_warp(bar_wfull + 8 * st, ph, flags)) { ok = false; break; }
                    ptx::tc_fence_after_sync();
                    const uint32_t a_lo = a_lo0 + s * a_step, w_lo = w_lo0 + st * w_step;
                    const int nks = c == p.kc - 1 ? p.ksteps_last : 4;
                    if (leader) {
                        if (c == 0) ptx::mma_i8_pair<false>(d_tmem, d_128 | (uint64_t)a_lo, d_128 | (uint64_t)w_lo, idesc);
                        else ptx::mma_i8_pair<true>(d_tmem, d_128 | (uint64_t)a_lo, d_128 | (uint64_t)w_lo, idesc);
#pragma unroll
                        for (int ks = 1; ks < 4; ++ks)
                            if (ks < nks)
                                ptx::mma_i8_pair<true>(d_tmem, d_128 | (uint64_t)(a_lo + 2 * ks), d_128 | (uint64_t)(w_lo + 2 * ks), idesc);
                        ptx::mma_commit_pair(bar_wempty + 8 * st);
                        if (last) ptx::mma_commit_pair(bar_aempty + 8 * s);
                    }
                    if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
                }
                if (!ok) break;
                // the bias step: the constant block of 1s and 127s against the tile's digits
                if (!tc::wait_bar_warp(bar_wfull + 8 * st, ph, flags)) { ok = false; break; }
                ptx::tc_fence_after_sync();
                if (leader) {
                    ptx::mma_i8_pair<true>(d_tmem, ac_desc, d_32 | (uint64_t)(w_lo0 + st * w_step), idesc);
                    ptx::mma_commit_pair(bar_wempty + 8 * st);
                    ptx::mma_commit_pair(bar_tfull + 8 * acc);
                }
                if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
                if (last) n0 += (uint32_t)p.kc;
                if (++ct == p.n_ctiles) ct = 0;
            }
            // the second CTA's read-outs arrive here
            for (int e = 0; e < 2 && ok; ++e, ++k)
                ok = tc::wait_bar_warp(bar_tempty + 8 * ((uint32_t)k & 1u), (((uint32_t)k >> 1) & 1u) ^ 1u, flags);
            // nothing of the pair's MMAs is outstanding (the second CTA learns of it at the teardown)
            if (leader) ptx::mma_commit_own(bar_drain);
            const unsigned long long t0 = ptx::globaltimer();
            while (!ptx::mbar_try_wait(bar_drain, 0) && ptx::globaltimer() - t0 < tc::kWaitLimitNs) {}
        }
        __syncwarp();
    } else {
        // ---- epilogue ---------------------------------------------------------------------------------
        // Four groups of four warps: group grp takes the pieces grp, grp + 4 of 32 columns of every unit.
        const int q = warp & 3, grp = (warp - 2) >> 2;
        uint8_t *slab = smem + p.off_out + (size_t)(warp - 2) * kSlabBytes;
        uint8_t *my_row = slab + lane * kEpiCols;
        const uint32_t slab_addr = ptx::smem_u32(slab);
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t tempty = ptx::map_to_rank(bar_tempty, 0);
        int mt = mt0, ct = ct0;
        for (int k = 0; k < n_units; ++k) {
            const uint32_t acc = (uint32_t)k & 1u, ph = ((uint32_t)k >> 1) & 1u;
            const int row0 = mt * 256 + (int)rank * 128 + q * 32, pieces = width(ct) / (int)kEpiCols;
            if (!tc::wait_bar<true>(bar_cfull + 8 * acc, ph, flags)) break;
            if (!tc::wait_bar<true>(bar_tfull + 8 * acc, ph, flags)) break;
            ptx::tc_fence_after_sync();
            // the accumulator is free for the MMAs once every warp has read its last piece
            auto release = [&] {
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(tempty + 8 * acc);
            };
            if (grp >= pieces) release();
#pragma unroll 1
            for (int pc = grp; pc < pieces; pc += 4) {
                const int at = pc * (int)kEpiCols;
                const uint8_t *cst = smem + p.off_const + (acc * (uint32_t)p.nb + (uint32_t)(at / kNt)) * kConstBytes;
                const int *cm = reinterpret_cast<const int *>(cst) + (at & (kNt - 1));
                const int2 *cbs = reinterpret_cast<const int2 *>(cst + kNt * 4) + (at & (kNt - 1));
                const int *hdr = reinterpret_cast<const int *>(cst + kNt * 12);
                const int shmax = hdr[0];
                const bool other_clamp = hdr[3] != clamp_code(p.act_min, p.act_max);
                const bool bad = hdr[2] != 0 || other_clamp, fast = hdr[1] != 0 && !bad, last = pc + 4 >= pieces;
                if (other_clamp && lane == 0) raise_status(PROM_ERR_BAD_REQUANT);
                const uint32_t taddr = t_lane + acc * 256u + (uint32_t)at;
                // the previous store has read the slab
                ptx::bulk_wait_read0();
                __syncwarp();
                if (fast) {
                    uint32_t v[32];
                    ptx::tmem_ld_x32(taddr, v);
                    ptx::tmem_wait_ld();
                    if (last) release();
                    if (p.act_min == 0) tc::fast_piece<32, false>(v, cm, 1ll << (32 + shmax), shmax, my_row, true);
                    else tc::fast_piece<32, true>(v, cm, 1ll << (32 + shmax), shmax, my_row, true);
                } else {
                    if (!bad) tc::epi_exact_subtile<32>(32, p.act_min, p.act_max, taddr, cm, cbs, my_row, 0u);
                    if (last) release();
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && row0 < p.m && !bad) {
                    ptx::tma_store_2d(&ymap, ct * nt + at, row0, slab_addr);
                    ptx::bulk_commit();
                }
            }
            // the unit's constants are free for the unit after next
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_cempty + 8 * acc);
            if (++ct == p.n_ctiles) { ct = 0; ++mt; }
        }
        ptx::bulk_wait_read0();
    }

    // ---- teardown ---------------------------------------------------------------------------------
    // (neither CTA may go while the other can still reach its shared memory)
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 512u);
    }
}

}}  // namespace prom::wide
