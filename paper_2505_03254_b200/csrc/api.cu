// Host side of the C ABI (include/prom.h): argument checks, variant choice,
// launch planning, tensor-map creation, and the layer-sequence driver.
#include <cuda.h>
#include <cuda_runtime.h>

#include <array>
#include <atomic>
#include <map>
#include <cstdio>
#include <cmath>
#include <cstring>
#include <mutex>
#include <thread>
#include <unordered_map>
#include <vector>

#include "prom.h"
#include "prom_debug.h"

#include "common.cuh"
#include "hostutil.cuh"
#include "simple.cuh"
#include "tc.cuh"
#include "chain.cuh"
#include "smallk.cuh"
#include "addsub.cuh"
#include "actquant.cuh"
#include "depthwise.cuh"
#include "dwtc.cuh"
#include "wide.cuh"
#include "block.cuh"
#include "stack.cuh"
#include "quantize.cuh"
#include "peak.cuh"

namespace prom {

static std::atomic<uint64_t> g_launches{0};

struct DeviceInfo {
    int sms = 0;
    int smem_optin = 0;
    int smem_total = 0;   // shared memory per SM
    int dev = 0;
    bool ok = false;
};

static DeviceInfo query_device(int dev)
{
    DeviceInfo d;
    d.dev = dev;
    d.ok = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&d.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&d.smem_total, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess;
    return d;
}

// The current device's limits; asked of the driver once per device.  A call is a few microseconds of
// host time, so the look-up takes no lock once the entry is there.
static DeviceInfo device_info()
{
    constexpr int kDevices = 64;
    static DeviceInfo cache[kDevices];
    static std::once_flag once[kDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return DeviceInfo();
    if (dev < 0 || dev >= kDevices) return query_device(dev);
    std::call_once(once[dev], [dev] { cache[dev] = query_device(dev); });
    return cache[dev];
}

// ---- the layer as the host sees it -----------------------------------------------
struct Conv {
    const int8_t *x;
    long long m;        // output rows
    int cin, cout;
    RowMap map;         // how output rows find their input rows
    long long in_rows;  // rows of the input matrix
    const uint8_t *w;
    prom_requant rq;
    int8_t *y;
    cudaStream_t st;
    int pdl = tc::kPdlWait;    // how the kernel is chained to the previous one (tc.cuh: kPdl*, 0: plain launch)
    bool pdl_next = true;      // the next kernel of the stream may chain to this one
    const int8_t *res = nullptr;   // added to the output with int8 saturation (may be y)
};

static inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static prom_status check_requant(const prom_requant *rq)
{
    if (!rq || !rq->bias || !rq->mult || !rq->shift) return PROM_ERR_NULL;
    if (rq->act_min < -128 || rq->act_max > 127 || rq->act_min > rq->act_max)
        return PROM_ERR_BAD_REQUANT;
    return PROM_OK;
}

static prom_status check_conv(const int8_t *x, long long m, int cin, const uint8_t *w, int cout,
                              const prom_requant *rq, const int8_t *y)
{
    if (!x || !w || !y) return PROM_ERR_NULL;
    prom_status s = check_requant(rq);
    if (s != PROM_OK) return s;
    if (m < 0 || cin < 1 || cin > 4096 || cout < 1 || cout > 4096) return PROM_ERR_SHAPE;
    if (m > (1ll << 40)) return PROM_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(w) || !aligned16(y)) return PROM_ERR_ALIGN;
    return PROM_OK;
}

static int grid_for(long long work_items, int threads, int sms)
{
    long long blocks = (work_items + threads - 1) / threads;
    long long cap = (long long)sms * 16;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

// With PROM_VERBOSE set in the environment the CUDA error behind a PROM_ERR_CUDA goes to stderr.
static prom_status cuda_status(cudaError_t e)
{
    if (e == cudaSuccess) return PROM_OK;
    static const bool verbose = getenv("PROM_VERBOSE") != nullptr;
    if (verbose) fprintf(stderr, "prom: CUDA error %d: %s\n", (int)e, cudaGetErrorString(e));
    return PROM_ERR_CUDA;
}

// Launch configuration of a kernel that may be chained to its predecessor in the stream with
// programmatic dependent launch (attr must outlive the launch call).
static void fill_launch_cfg(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int grid, int threads, size_t smem,
                            cudaStream_t st, bool pdl)
{
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    if (pdl) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
}

// ---- naive -------------------------------------------------------------------------------
static prom_status launch_naive(const Conv &c, int32_t *acc_out)
{
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    const int threads = 256;
    int grid = grid_for(c.m * c.cout, threads, d.sms);
    naive_conv_kernel<<<grid, threads, 0, c.st>>>(c.x, c.m, c.cin, c.map, c.w, c.cout, c.rq.bias,
                                                  c.rq.mult, c.rq.shift, c.rq.act_min,
                                                  c.rq.act_max, acc_out ? nullptr : c.y, acc_out,
                                                  acc_out ? nullptr : c.res);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

// ---- tensor-core variant: planning --------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) ==
                cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

struct TcPlan {
    tc::Params p;
    CUtensorMap xmap, ymap, tmap;
    int grid = 0;
    int per_sm = 2;        // CTAs of the launch that share an SM (picks the kernel build)
    size_t smem = 0;
    double est_us = 0;
};

// Tuning override (0 = automatic), set by prom_debug_tc_plan.
struct TcTune { int fold, nt, groups, occ, stages; };
static TcTune g_tune = {0, 0, 0, 0, 0};
// Overrides for single shapes (m, cin, cout, input stride), set by prom_debug_tc_plan_shape;
// they take precedence over g_tune for that shape.
static std::mutex g_shape_tune_mu;
static std::map<std::array<long long, 4>, TcTune> g_shape_tune;

// Whether any override is set (the look-up below takes a lock).
static std::atomic<bool> g_tuned{false};

static TcTune tune_for(long long m, int cin, int cout, int stride)
{
    if (!g_tuned.load()) return TcTune{0, 0, 0, 0, 0};
    std::lock_guard<std::mutex> lk(g_shape_tune_mu);
    auto it = g_shape_tune.find({m, cin, cout, stride});
    return it == g_shape_tune.end() ? g_tune : it->second;
}

// Depth-first execution of parts of a sequence, set by prom_debug_seq_chain.  Off unless asked
// for: on the network the library is timed on it is slower than one launch per layer.
static std::atomic<int> g_seq_chain{0};
// Every second layer of a sequence walks its row tiles from the last to the first, so that it
// reads first what the layer before wrote last (still in L2 when the tensor is larger than L2:
// 0.3220 -> 0.3196 ms per step on the timed network).  On unless prom_debug_seq_order(0).
static std::atomic<int> g_seq_snake{1};

static int round_up(int v, int a) { return (v + a - 1) / a * a; }

// Outputs up to about this size stay in L2 (126 MB) until they are complete.
constexpr double kL2Bytes = 0.8e8;

// Edges per row between subtiles that are written far apart in time, where subtiles are not whole 32-byte sectors:
// about half of them split one.  (One CTA that shares a tile's load among its subtiles writes both sides at once.)
static int torn_edges(const tc::Params &p)
{
    return p.n_sub > 1 && p.nt % 32 && (p.groups > 1 || !p.share_x) ? p.n_sub : 0;
}

// What a plan is for: kPlanSingle (one call: the kernel builds its operands itself), kPlanDynamic (the dynamic
// layer: no row folding, a folded row could straddle two samples) or
// kPlanPrepared (a layer of a sequence, whose operands tc_prep_kernel builds once)
// kPlanOdd, added to kPlanSingle or kPlanPrepared (the automatic choice of calls and sequences): an odd number of
// rows that have to be folded in pairs is taken too, the last row as a tile of its own (PROM_VARIANT_TC
// refuses such a shape), and small layers may have subtiles of any multiple of 8
// kPlanRes, added to kPlanSingle: a tensor is added to the output
enum { kPlanSingle = 0, kPlanDynamic = 1, kPlanPrepared = 2, kPlanOdd = 4, kPlanRes = 8 };

// Everything of a plan that follows from (fold, nt, groups, occ); false when it does not fit.
static bool tc_fill_plan(long long m, int cin, int cout, const RowMap &map, const DeviceInfo &d,
                         int fold, int nt, int groups, int occ, int want_stages, TcPlan &pl,
                         int cw_max = 128, int direct = 0, bool tail = false, int use = kPlanPrepared)
{
    tc::Params &p = pl.p;
    memset(&p, 0, sizeof(p));
    const int kf = cin * fold, nf = cout * fold;
    if (kf > 4096 || nf % nt) return false;
    const int n_sub = nf / nt;
    if (n_sub % groups) return false;
    // tensor-map stores want rows and subtiles of whole 16-byte pieces; a small layer may store its rows in
    // 8-byte pieces instead, which lets it use more than one channel group (720 -> 120 on 441 rows)
    const bool rows_8 = n_sub > 1 && ((nt & 15) || (nf & 15));
    if (rows_8 && (!(use & kPlanOdd) || direct || (nt & 7) || m * cout > 1500000)) return false;
    if (n_sub == 1 && (nt & 7)) return false;
    const int subs = n_sub / groups;
    const int nt_pad = round_up(nt, 16);
    if (nt_pad > 256) return false;
    const int cw = kf <= 32 ? 32 : (kf <= 64 || cw_max <= 64 ? 64 : 128);
    const int kc = (kf + cw - 1) / cw;

    // tile rows
    int tm = 128, x3d = 0, box_r = 0;
    if (map.stride != 1) {
        if (fold != 1 || map.wo > 128) return false;
        box_r = 128 / map.wo;
        long long lines = m / map.wo;          // batch * ho
        if (box_r > lines) box_r = (int)lines;
        if (box_r > 256) box_r = 256;
        tm = box_r * map.wo;
        x3d = 1;
    }
    const long long rows = m / fold;
    if ((nf & 15) && (tm & 1)) return false;     // slabs of the 1-D store start on 16-byte granules
    const long long n_mtiles = (rows + tm - 1) / tm + (tail ? 1 : 0);
    if (rows + 256 >= (1ll << 31)) return false;   // row coordinates are 32-bit in the kernel

    // tensor memory: the CTAs of an SM share its 512 columns
    // occ 1: one CTA with all of the SM; occ 2: two CTAs; occ 3: one CTA on half an SM, leaving
    // the other half to the next kernel's prologue; occ 4: three CTAs
    const int share = occ == 1 ? 1 : (occ == 4 ? 3 : 2);
    const int tmem_cols = share == 1 ? 512 : (share == 2 ? 256 : 128);
    if (2 * nt_pad > tmem_cols) return false;
    // accumulator ring: an even length, so that each of the two epilogue groups keeps to its own
    // accumulators
    if (tmem_cols / nt_pad < 2) return false;
    const int nbuf = tmem_cols / nt_pad >= 4 ? 4 : 2;

    // outputs straight from registers: rows and subtiles of whole 32-byte sectors (a partial sector costs
    // L2 a read-modify-write); three CTAs per SM have too few registers for it
    if (direct && (nt % 32 || nf % 32 || occ == 4 || tail)) return false;
    const int ncols = subs * nt_pad;
    const size_t stage_bytes = (size_t)128 * cw;
    const size_t w_bytes = (size_t)subs * kc * nt_pad * cw;
    const size_t wbias_bytes = (size_t)subs * nt_pad * 32;
    const size_t out_bytes = direct ? 0 : (size_t)tc::kEpiWarps * 32 * nt;
    const size_t fixed = w_bytes + wbias_bytes + tc::kAConstBytes + round_up((int)out_bytes, 128) +
                         (size_t)ncols * 12 + 16 + 256 + tc::kLuts * 1024 + 256 + 1024 /* alignment slack */;
    const size_t budget = share == 1 ? (size_t)d.smem_optin
                                     : (size_t)((d.smem_total - share * 1024) / share);
    if (budget > (size_t)d.smem_optin || fixed + 2 * stage_bytes > budget) return false;
    int stages = (int)((budget - fixed) / stage_bytes);
    const int share_x = (kc == 1 && subs > 1) ? 1 : 0;
    int cap = share_x ? 4 : (kc >= 4 ? tc::kMaxStages : 6);
    if (want_stages > 0) cap = want_stages;
    if (stages > cap) stages = cap;
    if (stages > tc::kMaxStages) stages = tc::kMaxStages;
    if (stages < 2) return false;
    // the packed weights of the CTA are copied into the activation stages before these are used
    {
        const size_t rowb = (size_t)(cin + 3) / 4;
        const size_t packed = fold > 1 ? (size_t)cout * rowb : (size_t)subs * nt * rowb;
        if (packed > (size_t)stages * stage_bytes) return false;
    }

    p.m_rows = rows; p.tail = tail ? 1 : 0; p.k0 = cin; p.n0 = cout; p.fold = fold; p.kf = kf; p.nf = nf;
    p.tm = tm; p.n_mtiles = (int)n_mtiles; p.nt = nt; p.nt_pad = nt_pad;
    p.n_sub = n_sub; p.groups = groups; p.subs_per_cta = subs;
    p.cw = cw; p.kc = kc;
    p.ksteps_last = (kf - (kc - 1) * cw + 31) / 32;
    p.stages = stages; p.nbuf = nbuf; p.tmem_cols = tmem_cols;
    p.share_x = share_x;
    p.direct = direct;
    p.store_2d = rows_8 ? 2 : (n_sub > 1 && !direct ? 1 : 0);
    p.x3d = x3d; p.box_r = box_r;
    p.tx_bytes = x3d ? (uint32_t)(cw * map.wo * box_r) : (uint32_t)stage_bytes;

    // shared-memory layout; [off_w, off_hdr + 16) is the CTA's prepared image
    uint32_t off = (uint32_t)(stages * stage_bytes);
    p.off_w = off; off += (uint32_t)w_bytes;
    p.off_wbias = off; off += (uint32_t)wbias_bytes;
    p.off_mult = off; off += (uint32_t)ncols * 4;
    p.off_bs = off; off += (uint32_t)ncols * 8;
    p.off_hdr = off; off += 16;
    p.image_bytes = off - p.off_w;
    p.image_stride = (p.image_bytes + 255u) & ~255u;
    off = (off + 255u) & ~255u;
    p.off_aconst = off; off += tc::kAConstBytes;
    p.off_out = off; off += (uint32_t)round_up((int)out_bytes, 128);
    p.off_lut = off; off += tc::kLuts * 1024;
    p.off_bars = off; off += 256;
    pl.smem = (size_t)off + 1024;
    if (occ == 1 && pl.smem * 2 + 2048 <= (size_t)d.smem_total)
        pl.smem = (size_t)d.smem_total / 2;       // keep a second CTA (and its TMEM request) off the SM
    if (pl.smem > (size_t)d.smem_optin) return false;

    const int per_sm = occ == 2 ? 2 : (occ == 4 ? 3 : 1);
    pl.per_sm = per_sm;
    const long long slots = (long long)d.sms * per_sm;
    long long workers = slots / groups;
    if (workers < 1) workers = 1;
    if (workers > n_mtiles) workers = n_mtiles;
    pl.grid = (int)(workers * groups);

    // Rough time model (microseconds), used only to rank candidate plans; the constants come
    // from timing the kernel on a B200.  A CTA pays a start-up that grows with the operands it
    // brings in, then streams its units at the rate the epilogue warps sustain, and ends with
    // the latency of its last unit (one warp draining nt columns, then the store).
    const double rounds = (double)((n_mtiles + workers - 1) / workers);
    const double ctas_per_sm = (double)pl.grid / d.sms < 1.0 ? 1.0
                               : ((double)pl.grid / d.sms > per_sm ? per_sm : (double)pl.grid / d.sms);
    const double epi_rate = 36e3 / ctas_per_sm;              // outputs per microsecond per CTA
    // an SM takes 58 bytes per clock from L2 (the copy-rate probe): 110 KB per microsecond
    const double load_rate = 110e3 / ctas_per_sm;            // bytes per microsecond per CTA
    // Staged subtile widths with a straight-line epilogue (tc.cuh: epi_fast_fixed); any other width that
    // splits a row runs the looped epilogue, measured ~1 us per layer slower at 128 columns.
    const bool straight = nt == 96 || nt == 64 || nt == 48 || nt == 32 || nt == 80;
    // What is written beyond L2, a share of the output that grows from nothing.  There a sector that torn_edges()
    // splits is written in two pieces that no longer meet, about three sectors more to move per edge (with a residual
    // its reads bring the sector into L2).  And where a unit is short (one K chunk of at most 64 bytes), stores from
    // registers, which do not run beside the next unit, cost more than staged ones (852992 rows, 16 -> 576: 157.0 us
    // direct in 128 columns, 139.4 staged in 96; but 478512 rows, 120 -> 960: 164.5 and 193.6).
    const bool res = (use & kPlanRes) != 0;
    const double out_all = (double)m * cout, beyond = out_all > kL2Bytes ? out_all - kL2Bytes : 0.0;
    const double t_torn = res ? 0.0 : beyond / cout * torn_edges(p) * 96.0 / 5.5e6;
    double epi_cost = direct ? 1.0 + (kf <= 64 ? 0.4 : 0.0) * beyond / out_all
                             : (straight ? 1.0 : (n_sub > 1 ? 1.5 : (nt <= 96 ? 1.0 : 1.15)));
    // A residual: its bytes are held in registers beside direct stores (which one CTA per SM does not hide), and for
    // the first 48 columns of a staged slab; those of the others are asked for once the accumulator is there, 25 ns a
    // column (781600 rows, 240 -> 320: 185.2 us direct in 64 columns, 464.0 staged in 160).
    if (res) epi_cost *= direct ? (occ == 1 ? 1.6 : 1.2) : 1.4;
    const double t_late = res && !direct && nt > 48 ? 0.025 * (nt - 48) : 0.0;
    const double t_epi = (double)tm * nt / epi_rate * epi_cost + t_late;
    const double t_load = (double)kc * tm * (kf < cw ? kf : cw) / load_rate;
    // Direct outputs want whole 64-column pieces: half of the stores of a last piece of 32 are short, which
    // shows once L2 is busy (16 -> 96 at 1.6 M rows 53.9 us against 46.3 staged, 64 -> 384 at 25088 rows 6.6
    // against 6.1; at 1176 rows, 160 -> 960, 4.3 against 4.8).  A bulk store runs beside the next unit, a
    // direct one does not, so several units per CTA lose a little of what one gains.
    const bool short_piece = direct && nt % 64 && nt > 32;
    const double unit = short_piece ? 1.15 : (direct && rounds * subs > 1 ? 0.9 : 0.8) + (rows_8 ? 0.3 : 0.0);
    // 0.8 us per unit for the hand-overs around it (barrier waits, fences, store issue): fitted to
    // plans timed inside the chained step (32 -> 192 and 64 -> 384 prefer 96-column subtiles in
    // fewer channel groups to 64-column ones)
    const double t_first = (t_epi > t_load ? t_epi : t_load) + unit;
    const double t_next = share_x ? t_epi + unit : t_first;
    // (a single call's CTAs expand their operands themselves: 18816 rows, 64 -> 1280 take 13.4 us with 80 columns per
    // CTA and 18.3 with 640)
    const double startup = 1.2 + (double)p.image_bytes / 80e3 * ctas_per_sm * ((use & 3) == kPlanSingle ? 1.5 : 1.0);
    const double fill = 1.0 + 0.1 * kc;                      // first load, first MMA
    // Draining the last accumulator, store.  A direct store saves the hand-over to the bulk-copy unit: at
    // 392 rows, 64 -> 384 takes 3.1 / 3.4 / 3.9 us with 32 / 64 / 128 columns against 3.4 / 3.6 / 4.5 staged
    // (and 3.5 with 16), 384 -> 64 3.8 against 4.2.
    const double last = direct && !(short_piece && m * cout > 6000000) ? 0.35 * ((nt + 31) / 32) + 0.5 : 0.45 * ((nt + 31) / 32) + 0.8;
    const double t_cta = startup + fill + rounds * (t_first + (subs - 1) * t_next) + last +
                         (occ == 1 ? 2.5 : 0.0);   // a CTA that fills its SM keeps the next kernel out
    // X is read once per unit, or per channel group where one load serves all subtiles of the tile; all readings but the
    // first come from L2.
    const int readings = share_x ? groups : n_sub;
    const double t_mem = ((double)m * cin * (1.0 + 0.1 * (readings - 1)) + (res ? 2.0 : 1.0) * out_all) / 5.5e6;
    // The constants above were fitted to 3892 calls drawn over the networks' widths and spatial sizes (plain, linear,
    // with a residual, prepared, dynamic), every plan timed: the chosen plan takes 1.5 to 2 % more than the best on
    // average (dynamic layers 4 %).
    pl.est_us = (t_cta > t_mem ? t_cta : t_mem) + t_torn;
    return true;
}

// Picks fold, subtile width, channel groups and occupancy.  Returns false when
// the tensor-core variant cannot run this shape.  use: kPlan*
static bool tc_search_plan(long long m, int cin, int cout, const RowMap &map, const DeviceInfo &d,
                           int use, TcPlan &best)
{
    const bool dyn = (use & 3) == kPlanDynamic, odd_ok = (use & kPlanOdd) != 0;
    bool tail = false;
    if (m <= 0 || (cin & 7) || (cout & 7)) return false;
    const TcTune tn = tune_for(m, cin, cout, map.stride);
    int fold = 1;
    if (map.stride == 1) {
        // Rows that are not 16-byte multiples cannot be described to TMA: two rows are folded into
        // one.  On the output side that is only needed when the row does not fit one subtile
        // (a slab of 32 whole rows is then one contiguous, 16-byte aligned range of Y anyway).
        if ((cin & 15) || ((cout & 15) && cout > 256 && (m % 2 == 0 || odd_ok))) fold = 2;
        tail = m % fold != 0;
        if (tail && !odd_ok) return false;
        while (!tail && fold * 2 <= 8 && fold * 2 * cin <= 128 && fold * 2 * cout <= 128 &&
               m % (fold * 2) == 0)
            fold *= 2;
        // rows of fewer than 32 bytes make poor TMA boxes (measured on the 16 -> 96 layer: 3 us
        // of 58): fold once more whatever the width, where the larger block-diagonal weights
        // are expanded once per sequence and not by every CTA
        // (a single call expands them in every CTA, which pays when the CTA then has many tiles)
        // (and unless the doubled width has no subtile with a straight-line epilogue: 16 -> 112 at 852074 rows takes
        // 41.8 us folded against 39.2)
        const int twice = cout * fold * 2;
        const bool many = m >= 128ll * 16 * 2 * d.sms && (twice % 48 == 0 || twice % 64 == 0 || twice % 80 == 0);
        if (!tail && ((use & 3) == kPlanPrepared || many) && cin * fold < 32 && fold * 2 <= 8 && m % (fold * 2) == 0) fold *= 2;
    }
    if (dyn) {
        if ((cin & 15) || ((cout & 15) && cout > 256)) return false;
        fold = 1;
    }
    if (tn.fold > 0) fold = tn.fold;
    if (fold < 1 || fold > 8) return false;
    if (m % fold && !(tail && fold == 2)) return false;
    if (fold == 1) tail = false;
    const int nf = cout * fold;
    bool found = false;
    for (int nt = 8; nt <= 256 && nt <= nf; nt += 8) {
        if (nf % nt) continue;
        if (tn.nt > 0 && nt != tn.nt) continue;
        const int n_sub = nf / nt;
        for (int groups = 1; groups <= n_sub; ++groups) {
            if (n_sub % groups) continue;
            if (tn.groups > 0 && groups != tn.groups) continue;
            for (int occ = 4; occ >= 1; --occ) {
                if (tn.occ > 0 && occ != tn.occ) continue;
                if (dyn && occ > 2) continue;
                if (tn.occ == 0 && occ >= 3) continue;      // only on request for now
                for (int direct = dyn ? 0 : 1; direct >= 0; --direct) {
                    TcPlan pl;
                    if (!tc_fill_plan(m, cin, cout, map, d, fold, nt, groups, occ, tn.stages, pl, 128, direct, tail, use))
                        continue;
                    if (!found || pl.est_us < best.est_us) { best = pl; found = true; }
                }
            }
        }
    }
    return found;
}


// The search above costs tens of microseconds; its result depends only on the shape, the
// device and the tuning override, so it is remembered: per process, and the last plans a thread has
// used in a small table of its own in front of that, so that a repeated call takes no lock.
typedef std::array<long long, 15> PlanKey;
struct PlanEntry { PlanKey key; bool ok; TcPlan pl; };

static void tc_find_plan(long long m, int cin, int cout, const RowMap &map, const DeviceInfo &d, int use,
                         const PlanKey &key, PlanEntry &out)
{
    static std::mutex mu;
    static std::map<PlanKey, PlanEntry> cache;
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it == cache.end()) {
        PlanEntry e;
        e.key = key;
        e.ok = tc_search_plan(m, cin, cout, map, d, use, e.pl);
        if (cache.size() > 4096) cache.clear();
        it = cache.emplace(key, e).first;
    }
    out = it->second;
}

static bool tc_shape_plan(long long m, int cin, int cout, const RowMap &map, const DeviceInfo &d,
                          TcPlan &best, int use = kPlanSingle)
{
    constexpr int kRecent = 128;
    static thread_local std::vector<PlanEntry> recent(kRecent, PlanEntry{PlanKey{}, false, TcPlan()});
    const TcTune tn = tune_for(m, cin, cout, map.stride);
    const PlanKey key = {m, cin, cout, map.stride, map.ho, map.wo, map.hin, map.win,
                         tn.fold, tn.nt, tn.groups, tn.occ, tn.stages, d.dev, use + 1};
    const unsigned long long h = ((unsigned long long)m * 0x9E3779B1u + (unsigned)cin * 0x85EBCA6Bu +
                                  (unsigned)cout * 0xC2B2AE35u + (unsigned)(map.stride * 16 + use) * 0x27D4EB2Fu);
    PlanEntry &e = recent[(h ^ (h >> 17)) & (kRecent - 1)];
    if (e.key != key) tc_find_plan(m, cin, cout, map, d, use, key, e);
    if (e.ok) best = e.pl;
    return e.ok;
}

static bool tc_make_maps(const Conv &c, TcPlan &pl)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const tc::Params &p = pl.p;
    const CUtensorMapSwizzle sw = p.cw == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                  : (p.cw == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    CUresult r;
    if (!p.x3d) {
        cuuint64_t dims[2] = {(cuuint64_t)p.kf, (cuuint64_t)(p.m_rows > 0 ? p.m_rows : 1)};
        cuuint64_t strides[1] = {(cuuint64_t)p.kf};
        cuuint32_t box[2] = {(cuuint32_t)p.cw, 128};
        cuuint32_t es[2] = {1, 1};
        r = enc(&pl.xmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(c.x), dims, strides,
                box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        // [channel][wo, step stride*cin][batch*ho, step stride*win*cin]
        const RowMap &mp = c.map;
        cuuint64_t dims[3] = {(cuuint64_t)c.cin, (cuuint64_t)mp.wo, (cuuint64_t)(c.m / mp.wo)};
        cuuint64_t strides[2] = {(cuuint64_t)mp.stride * c.cin,
                                 (cuuint64_t)mp.stride * mp.win * c.cin};
        cuuint32_t box[3] = {(cuuint32_t)p.cw, (cuuint32_t)mp.wo, (cuuint32_t)p.box_r};
        cuuint32_t es[3] = {1, 1, 1};
        r = enc(&pl.xmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t *>(c.x), dims, strides,
                box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return false;
    if (p.store_2d == 1) {
        cuuint64_t dims[2] = {(cuuint64_t)p.nf, (cuuint64_t)(p.m_rows > 0 ? p.m_rows : 1)};
        cuuint64_t strides[1] = {(cuuint64_t)p.nf};
        cuuint32_t box[2] = {(cuuint32_t)p.nt, 32};
        cuuint32_t es[2] = {1, 1};
        r = enc(&pl.ymap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, c.y, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return false;
    } else {
        pl.ymap = pl.xmap;      // unused by the kernel
    }
    pl.tmap = pl.xmap;          // unused by the kernel without a tail
    if (p.tail) {
        // the last row alone: columns past cin and the box's other rows arrive as zeros
        cuuint64_t dims[2] = {(cuuint64_t)p.k0, 1};
        cuuint64_t strides[1] = {(cuuint64_t)p.kf};
        cuuint32_t box[2] = {(cuuint32_t)p.cw, 128};
        cuuint32_t es[2] = {1, 1};
        r = enc(&pl.tmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(c.x) + p.m_rows * p.kf, dims, strides,
                box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return false;
    }
    return true;
}

static prom_status tc_set_attr(const DeviceInfo &d)
{
    // once per device: the limit is an attribute of the (function, device) pair
    static std::atomic<unsigned long long> done{0};
    const unsigned long long bit = d.dev >= 0 && d.dev < 64 ? 1ull << d.dev : 0ull;
    if (done.load(std::memory_order_acquire) & bit) return PROM_OK;
    cudaError_t e = raise_smem_limit(tc::tc_conv_kernel<2>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<3>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 1>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 2>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 4>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 3>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 0, true>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 3, true>, d.smem_optin);
    if (e == cudaSuccess) e = raise_smem_limit(tc::tc_conv_kernel<2, 4, true>, d.smem_optin);
    if (e != cudaSuccess) return PROM_ERR_CUDA;
    done.fetch_or(bit, std::memory_order_release);
    return PROM_OK;
}

// Fills in the pointers of a planned layer (image: prepared operands, or null).
static void tc_bind(const Conv &c, TcPlan &pl, uint8_t *image)
{
    tc::Params &p = pl.p;
    p.w_packed = c.w; p.bias = c.rq.bias; p.mult = c.rq.mult; p.shift = c.rq.shift;
    p.act_min = c.rq.act_min; p.act_max = c.rq.act_max; p.y = c.y; p.pdl = c.pdl;
    p.pdl_next = c.pdl_next ? 1 : 0;
    p.image = image;
    p.res = c.res;
}

static prom_status tc_launch_planned(const Conv &c, TcPlan &pl, int mode = 0)
{
    if (!tc_make_maps(c, pl)) return PROM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, pl.grid, tc::kThreads, pl.smem, c.st, c.pdl != 0);
    cudaError_t e;
    if (mode == 1) e = cudaLaunchKernelEx(&cfg, tc::tc_conv_kernel<2, 1>, pl.xmap, pl.ymap, pl.tmap, pl.p);
    else if (mode == 2) e = cudaLaunchKernelEx(&cfg, tc::tc_conv_kernel<2, 2>, pl.xmap, pl.ymap, pl.tmap, pl.p);
    else {
        const bool full_range = pl.p.act_min == -128 && pl.p.act_max == 127;
        auto *kernel = pl.p.direct ? (c.res ? tc::tc_conv_kernel<2, 3, true>
                                            : (full_range ? tc::tc_conv_kernel<2, 4, true> : tc::tc_conv_kernel<2, 0, true>))
                                   : (c.res ? tc::tc_conv_kernel<2, 3>
                                            : (full_range ? tc::tc_conv_kernel<2, 4>
                                               : pl.per_sm == 3 ? tc::tc_conv_kernel<3> : tc::tc_conv_kernel<2, 0>));
        e = cudaLaunchKernelEx(&cfg, kernel, pl.xmap, pl.ymap, pl.tmap, pl.p);
    }
    ++g_launches;
    return cuda_status(e);
}

// Adds a planned layer with an image to a preparation launch.
static void prep_add(tc::PrepTable &t, const tc::Params &p, int &ctas, size_t &smem)
{
    tc::PrepLayer &q = t.layer[t.n];
    q.w_packed = p.w_packed; q.bias = p.bias; q.mult = p.mult; q.shift = p.shift;
    q.image = p.image; q.image_stride = p.image_stride;
    q.off_wbias = p.off_wbias - p.off_w; q.off_mult = p.off_mult - p.off_w;
    q.off_bs = p.off_bs - p.off_w; q.off_hdr = p.off_hdr - p.off_w;
    q.k0 = p.k0; q.n0 = p.n0; q.fold = p.fold; q.kf = p.kf; q.nf = p.nf; q.nt = p.nt; q.nt_pad = p.nt_pad;
    q.groups = p.groups; q.subs = p.subs_per_cta; q.cw = p.cw; q.kc = p.kc; q.ksteps_last = p.ksteps_last;
    q.direct = p.direct; q.act_min = p.act_min; q.act_max = p.act_max;
    const int pieces = p.subs_per_cta * p.kc * p.nt_pad * (p.cw >> 4);
    q.parts = (pieces + tc::kPrepPieces - 1) / tc::kPrepPieces;
    t.first[t.n] = ctas;
    ctas += p.groups * q.parts;
    t.first[++t.n] = ctas;
    const size_t bytes = (size_t)p.subs_per_cta * p.nt_pad * sizeof(int2);
    if (bytes > smem) smem = bytes;
}

static size_t round256(size_t v) { return (v + 255) & ~(size_t)255; }

// ---- the row-resident variant for contraction-bound layers (wide.cuh) ----------------------------
// 0: the library's choice, 1: never, 2: whenever the shape allows it
static std::atomic<int> g_wide_mode{0};
static std::atomic<int> g_wide_nb{0};        // 0: the planner's choice; 1 or 2: forced (tests)

// Global scratch of the variant: the expanded weight matrix, bias digits, constants.
// (The handle of the per-thread default stream names a stream in every thread: the thread is part of the key there.)
struct WideKey {
    int dev;
    cudaStream_t st;
    std::thread::id thread;
    bool operator<(const WideKey &o) const
    {
        return dev != o.dev ? dev < o.dev : (st != o.st ? st < o.st : thread < o.thread);
    }
};
struct WideBuf { uint8_t *p = nullptr; size_t bytes = 0; };
static std::mutex g_wide_mu;
static std::map<WideKey, WideBuf> g_wide_cache;

static std::vector<uint8_t *> g_wide_retired;

// cudaMalloc that neither fails nor spoils a capture because a stream (this one or another thread's) is being captured.
static cudaError_t malloc_beside_capture(uint8_t **p, size_t bytes)
{
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaMalloc(reinterpret_cast<void **>(p), bytes);
    cudaThreadExchangeStreamCaptureMode(&mode);
    return e;
}

static size_t wide_buffer_size(size_t bytes)
{
    size_t want = 1 << 20;
    while (want < bytes) want *= 2;
    return want;
}

// A stream's buffer, for calls that run as they are made: in stream order, so that one buffer serves all of them.
// One that has become too small is kept until prom_shutdown(): earlier calls may still use it.  Sizes are powers of
// two, so a stream's buffers add up to less than twice its largest.  null: no memory.
static uint8_t *wide_scratch_for(cudaStream_t st, size_t bytes)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lk(g_wide_mu);
    WideBuf &b = g_wide_cache[WideKey{dev, st, st == cudaStreamPerThread ? std::this_thread::get_id() : std::thread::id()}];
    if (b.bytes < bytes) {
        const size_t want = wide_buffer_size(bytes);
        uint8_t *p = nullptr;
        if (malloc_beside_capture(&p, want) != cudaSuccess) return nullptr;
        if (b.p) g_wide_retired.push_back(b.p);
        b.p = p;
        b.bytes = want;
    }
    return b.p;
}

// A captured call runs whenever its graph does, on any stream and beside any other call, so it has a buffer of its own,
// which belongs to the graph: it becomes idle when the graph and all that was instantiated from it are gone, and serves
// a later capture.  (Mutex and table are never destroyed: the last graphs may go after this library's static objects.)
struct GraphBuf { int dev; size_t bytes; uint8_t *p; };
static std::mutex &graph_mu() { static std::mutex *m = new std::mutex; return *m; }
static std::vector<GraphBuf> &graph_idle() { static auto *v = new std::vector<GraphBuf>; return *v; }

static void CUDART_CB graph_buffer_idle(void *buf)       // (may call nothing of CUDA)
{
    GraphBuf *b = static_cast<GraphBuf *>(buf);
    std::lock_guard<std::mutex> lk(graph_mu());
    graph_idle().push_back(*b);
    delete b;
}

static uint8_t *graph_scratch_for(cudaStream_t st, size_t bytes)
{
    int dev = 0;
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaStreamGetCaptureInfo_v2(st, &status, nullptr, &graph, nullptr, nullptr) != cudaSuccess ||
        status != cudaStreamCaptureStatusActive || !graph)
        return nullptr;
    GraphBuf *b = new GraphBuf{dev, wide_buffer_size(bytes), nullptr};
    {
        std::lock_guard<std::mutex> lk(graph_mu());
        auto &idle = graph_idle();
        for (size_t i = 0; i < idle.size(); ++i)
            if (idle[i].dev == dev && idle[i].bytes == b->bytes) {
                b->p = idle[i].p;
                idle.erase(idle.begin() + i);
                break;
            }
    }
    if (!b->p && malloc_beside_capture(&b->p, b->bytes) != cudaSuccess) {
        delete b;
        return nullptr;
    }
    uint8_t *p = b->p;
    cudaUserObject_t owner = nullptr;
    if (cudaUserObjectCreate(&owner, b, graph_buffer_idle, 1, cudaUserObjectNoDestructorSync) != cudaSuccess) {
        graph_buffer_idle(b);
        return nullptr;
    }
    if (cudaGraphRetainUserObject(graph, owner, 1, cudaGraphUserObjectMove) != cudaSuccess) {
        cudaUserObjectRelease(owner, 1);
        return nullptr;
    }
    return p;
}

static void wide_release_cache()
{
    {
        std::lock_guard<std::mutex> lk(g_wide_mu);
        for (auto &kv : g_wide_cache)
            if (kv.second.p) cudaFree(kv.second.p);
        g_wide_cache.clear();
        for (uint8_t *p : g_wide_retired) cudaFree(p);
        g_wide_retired.clear();
    }
    std::lock_guard<std::mutex> lk(graph_mu());
    for (const GraphBuf &b : graph_idle()) cudaFree(b.p);
    graph_idle().clear();
}

struct WidePlan {
    wide::Params p;
    int grid;
    size_t smem;
    int k_pad;
};

// Pairs of CTAs that are resident at once, one CTA per SM (asked once per device: the query takes tens of
// microseconds).
static int wide_pairs(const DeviceInfo &d)
{
    static std::atomic<int> known[64];
    const bool keep = d.dev >= 0 && d.dev < 64;
    int n = keep ? known[d.dev].load() : 0;
    if (n == 0) {
        if (raise_smem_limit(wide::wide_conv_kernel, d.smem_optin) != cudaSuccess) return 0;
        cudaLaunchConfig_t cfg;
        fill_launch_cfg(cfg, nullptr, 2 * (d.sms / 2), wide::kThreads, (size_t)d.smem_optin, nullptr, false);
        if (cudaOccupancyMaxActiveClusters(&n, wide::wide_conv_kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        if (n > d.sms / 2) n = d.sms / 2;
        if (keep) known[d.dev].store(n);
    }
    return n;
}

// Shapes the variant takes: a plain matrix, whole 16-channel slices on both sides, K within the
// resident chunks.  `worth` says whether the library picks it by itself.
static bool wide_plan(const Conv &c, const DeviceInfo &d, WidePlan &pl, bool &worth)
{
    if (c.map.stride != 1 || c.res) return false;
    if ((c.cin & 15) || (c.cout & 15) || c.cin < wide::kChunk || c.cin > wide::kChunk * wide::kMaxKc) return false;
    if (c.cout < 64) return false;
    if (c.m >= (1ll << 31) - 256) return false;
    wide::Params &p = pl.p;
    memset(&p, 0, sizeof(p));
    p.m = c.m; p.cin = c.cin; p.cout = c.cout;
    p.kc = (c.cin + wide::kChunk - 1) / wide::kChunk;
    p.ksteps_last = (c.cin - (p.kc - 1) * wide::kChunk + 31) / 32;
    p.n_mtiles = (int)((c.m + 255) / 256);
    pl.k_pad = p.kc * wide::kChunk;
    // 256-channel column tiles; 128 (and 256 by number, up to Cin 512) only through prom_debug_tc_wide, for tests
    const int forced = g_wide_nb.load();
    if (forced == 2 && c.cin > 512) return false;
    const int nb = forced ? forced : 2;
    p.nb = nb;
    // shared memory: resident chunks, weight ring, constants, staging slabs, the bias step's A block, barriers
    const uint32_t a_bytes = (uint32_t)wide::kASlots * wide::kAChunkBytes, w_stage = (uint32_t)nb * (wide::kNt / 2) * wide::kChunk;
    const uint32_t const_bytes = ((uint32_t)(wide::kAccs * nb) * wide::kConstBytes + 1023u) & ~1023u;
    const uint32_t fixed = const_bytes + wide::kEpiWarps * wide::kSlabBytes + tc::kAConstBytes + 1024;
    const long long room = (long long)d.smem_optin - 1024 - a_bytes - fixed;
    int stages = (int)(room / w_stage);
    if (stages > wide::kMaxStages) stages = wide::kMaxStages;
    if (stages < 3) return false;
    p.stages = stages;
    p.n_ctiles = (c.cout + nb * wide::kNt - 1) / (nb * wide::kNt);
    p.off_w = a_bytes;
    p.off_aconst = p.off_w + (uint32_t)stages * w_stage;
    p.off_const = p.off_aconst + tc::kAConstBytes;
    p.off_out = p.off_const + const_bytes;
    p.off_bars = p.off_out + wide::kEpiWarps * wide::kSlabBytes;
    pl.smem = p.off_bars + 1024 + 1024;
    long long pairs = wide_pairs(d);
    if (pairs < 1) return false;
    if (pairs > (long long)p.n_mtiles * p.n_ctiles) pairs = (long long)p.n_mtiles * p.n_ctiles;
    pl.grid = (int)(2 * pairs);
    p.act_min = c.rq.act_min; p.act_max = c.rq.act_max;
    // Measured on B200, time as a share of the weight-resident kernel's (rows: 12544 / 50176 / 802816):
    //   Cin 960, Cout 1280: 0.65 0.54 0.47, 320: 0.97 0.79 0.69, 160: 0.80 0.81 0.83, 64: 0.82 0.92 0.97
    //   Cin 576, Cout 1280: 0.76 0.64 0.53, 320: 0.97 0.85 0.75, 160: 0.85 0.87 0.91, but 64: 0.93 0.96 1.20
    //   Cin 512, Cout 1280: 0.74 0.74 0.78, 240: 0.86 0.85 0.65, but 160: 0.86 0.94 1.02
    //   Cin 320, Cout 1280: 0.89 0.88 0.86, 320: 0.98 0.97 0.88, 256: 0.77 0.89 0.91, but 192: 0.86 0.95 1.08
    //   Cin 256, Cout 1280: 0.97 0.93 1.00, 320: 1.01 1.01 1.01
    // and on 6272 rows Cin 512, Cout 240 0.91, 1280 0.89, but Cin 320, Cout 720 1.11; on 3136 rows Cin 576,
    // Cout 320 0.95, 720 0.84, but 256 1.05.  Its one-multiply epilogue is for the clamps [0, 127] and [-128, 127].
    const long long rows_per_sm = c.m / d.sms;
    worth = ((rows_per_sm >= 80 && ((c.cin >= 320 && c.cout >= 256) || c.cin >= 960)) ||
             (rows_per_sm >= 40 && ((c.cin >= 512 && c.cout >= 240) || (c.cin >= 576 && c.cout >= 160))) ||
             (rows_per_sm >= 20 && c.cin >= 576 && c.cout >= 320)) &&
            (c.rq.act_min == 0 || c.rq.act_min == -128) && c.rq.act_max == 127;
    return true;
}

// The same question for operands prepared ahead of the call, which spares the weight-resident kernel more than
// this one (whose operands take a kernel of their own, 4 us).  Time as a share of the other's (rows: 12544 / 25088 /
// 401408): Cin 960, Cout 160: 0.76 0.92 0.87, 1280: 0.57 0.56 0.51; Cin 576, Cout 240: 0.85 0.74 0.49, but 160: 0.81
// 0.95 1.06; Cin 320, Cout 576: 0.99 0.95 0.97, 1280: 0.92 0.91 0.83, but 384: 1.11 1.06 0.91; Cin 192, Cout 1280:
// 1.01 0.99 1.00.  On 6272 rows Cin 960, Cout 320 0.99, 576 0.85, but Cin 576: 1.02 1.07; on 3136 rows Cin 576,
// Cout 960 0.97, 1280 0.82.  Other clamps, the 64-bit epilogue in both kernels: 0.67 to 1.0 from 25088 rows on (576 ->
// 240 1.15), on 6272 and 12544 rows 0.76 to 1.15.  (The size of the buffer is asked for without the clamp.)
static bool wide_prepared_worth(const Conv &c, const DeviceInfo &d)
{
    const long long rows_per_sm = c.m / d.sms;
    return (rows_per_sm >= 80 && ((c.cin >= 320 && c.cout >= 512) || (c.cin >= 576 && c.cout >= 240) ||
                                  (c.cin >= 960 && c.cout >= 160))) ||
           (rows_per_sm >= 40 && c.cin >= 960 && c.cout >= 320) ||
           (rows_per_sm >= 20 && c.cin >= 576 && c.cout >= 960);
}

// The kernel's operands in global memory: int8 weights, bias digits, constants.
static size_t wide_w8_bytes(const WidePlan &pl) { return (size_t)pl.p.n_ctiles * pl.p.nb * wide::kNt * pl.k_pad; }
static size_t wide_wbias_bytes(const WidePlan &pl) { return (size_t)pl.p.n_ctiles * pl.p.nb * wide::kWbiasBytes; }
static size_t wide_operand_bytes(const WidePlan &pl)
{
    return wide_w8_bytes(pl) + wide_wbias_bytes(pl) + round256((size_t)pl.p.n_ctiles * pl.p.nb * wide::kConstBytes);
}

static prom_status launch_wide_prep(const Conv &c, const WidePlan &pl, uint8_t *operands)
{
    wide::PrepParams pp;
    memset(&pp, 0, sizeof(pp));
    pp.cin = c.cin; pp.cout = c.cout; pp.k_pad = pl.k_pad; pp.w_packed = c.w;
    pp.bias = c.rq.bias; pp.mult = c.rq.mult; pp.shift = c.rq.shift;
    pp.act_min = c.rq.act_min; pp.act_max = c.rq.act_max; pp.signed_fast = 1;
    pp.w8 = reinterpret_cast<int8_t *>(operands); pp.wbias = operands + wide_w8_bytes(pl);
    pp.consts = pp.wbias + wide_wbias_bytes(pl);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, pl.p.n_ctiles * pl.p.nb * wide::kPrepParts, 256, 0, c.st, true);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, wide::wide_prep_kernel, pp);
    ++g_launches;
    return cuda_status(e);
}

static prom_status launch_wide_conv(const Conv &c, WidePlan &pl, uint8_t *operands)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return PROM_ERR_UNSUPPORTED;
    wide::Params &p = pl.p;
    const int blocks = p.n_ctiles * p.nb;           // of 128 channels
    uint8_t *wbias = operands + wide_w8_bytes(pl);
    p.consts = wbias + wide_wbias_bytes(pl);
    CUtensorMap xmap, wmap, bmap, ymap;
    cuuint32_t es[2] = {1, 1};
    {
        cuuint64_t dims[2] = {(cuuint64_t)c.cin, (cuuint64_t)c.m};
        cuuint64_t strides[1] = {(cuuint64_t)c.cin};
        cuuint32_t box[2] = {(cuuint32_t)wide::kChunk, 128};
        if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(c.x), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PROM_ERR_UNSUPPORTED;
    }
    {
        cuuint64_t dims[2] = {(cuuint64_t)pl.k_pad, (cuuint64_t)blocks * wide::kNt};
        cuuint64_t strides[1] = {(cuuint64_t)pl.k_pad};
        cuuint32_t box[2] = {(cuuint32_t)wide::kChunk, (cuuint32_t)(p.nb * wide::kNt / 2)};      // one CTA's half
        if (enc(&wmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, operands, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return PROM_ERR_UNSUPPORTED;
    }
    {
        cuuint64_t dims[2] = {32, (cuuint64_t)blocks * wide::kNt};
        cuuint64_t strides[1] = {32};
        cuuint32_t box[2] = {32, (cuuint32_t)(p.nb * wide::kNt / 2)};
        if (enc(&bmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, wbias, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PROM_ERR_UNSUPPORTED;
    }
    {
        cuuint64_t dims[2] = {(cuuint64_t)c.cout, (cuuint64_t)c.m};
        cuuint64_t strides[1] = {(cuuint64_t)c.cout};
        cuuint32_t box[2] = {wide::kEpiCols, 32};
        if (enc(&ymap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, c.y, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return PROM_ERR_UNSUPPORTED;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, pl.grid, wide::kThreads, pl.smem, c.st, true);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, wide::wide_conv_kernel, xmap, wmap, bmap, ymap, p);
    ++g_launches;
    return cuda_status(e);
}

static prom_status launch_wide(const Conv &c, WidePlan &pl)
{
    if (!encode_tiled_fn()) return PROM_ERR_UNSUPPORTED;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c.st, &cs) != cudaSuccess) {
        cudaGetLastError();
        return PROM_ERR_UNSUPPORTED;
    }
    uint8_t *scratch = cs == cudaStreamCaptureStatusNone ? wide_scratch_for(c.st, wide_operand_bytes(pl))
                                                         : graph_scratch_for(c.st, wide_operand_bytes(pl));
    if (!scratch) {             // no memory: the weight-resident kernel needs none
        cudaGetLastError();
        return PROM_ERR_UNSUPPORTED;
    }
    // Both launches as one: another thread's call on this stream must not put its operands between them.
    static std::mutex order;
    std::lock_guard<std::mutex> lk(order);
    const prom_status e = launch_wide_prep(c, pl, scratch);
    return e != PROM_OK ? e : launch_wide_conv(c, pl, scratch);
}

static prom_status launch_tc(const Conv &c, int use = kPlanSingle)
{
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    const int wide_mode = g_wide_mode.load();
    if (wide_mode != 1) {
        WidePlan wp;
        bool worth = false;
        if (wide_plan(c, d, wp, worth) && (worth || wide_mode == 2)) {
            const prom_status e = launch_wide(c, wp);
            if (e != PROM_ERR_UNSUPPORTED) return e;
        } else if (wide_mode == 2) {
            return PROM_ERR_UNSUPPORTED;
        }
    }
    TcPlan pl;
    if (!tc_shape_plan(c.m, c.cin, c.cout, c.map, d, pl, c.res ? use | kPlanRes : use)) return PROM_ERR_UNSUPPORTED;
    if (tc_set_attr(d) != PROM_OK) return PROM_ERR_CUDA;
    tc_bind(c, pl, nullptr);
    return tc_launch_planned(c, pl);
}

// ---- variant choice --------------------------------------------------------------------------
static prom_status run_conv(const Conv &c, prom_variant v)
{
    if (c.m == 0) return PROM_OK;
    // the residual is fused into the tensor-core and the naive kernels only
    if (c.res && (v == PROM_VARIANT_SMALLK || v == PROM_VARIANT_ADDSUB)) return PROM_ERR_UNSUPPORTED;
    switch (v) {
    case PROM_VARIANT_NAIVE: return launch_naive(c, nullptr);
    case PROM_VARIANT_TC: return launch_tc(c);
    case PROM_VARIANT_SMALLK: return smallk::launch(c.x, c.m, c.cin, c.map, c.w, c.cout, c.rq, c.y,
                                                    c.st, g_launches);
    case PROM_VARIANT_ADDSUB: return addsub::launch(c.x, c.m, c.cin, c.map, c.w, c.cout, c.rq, c.y,
                                                    c.st, g_launches);
    case PROM_VARIANT_AUTO: {
        const prom_status e = launch_tc(c, kPlanOdd);
        if (e != PROM_ERR_UNSUPPORTED) return e;
        if (!c.res && smallk::supported(c.cin, c.cout))
            return smallk::launch(c.x, c.m, c.cin, c.map, c.w, c.cout, c.rq, c.y, c.st, g_launches);
        return launch_naive(c, nullptr);
    }
    default: return PROM_ERR_UNSUPPORTED;
    }
}


// Shapes of a sequence; false when it does not chain.
struct SeqShape {
    std::vector<long long> m;      // output rows per layer
    std::vector<RowMap> map;
    std::vector<int> h, w;
};

static bool seq_shapes(const prom_layer *layers, int n, int batch, int h0, int w0, SeqShape &s)
{
    if (!layers || n < 1 || batch < 1 || h0 < 1 || w0 < 1) return false;
    int h = h0, w = w0;
    for (int i = 0; i < n; ++i) {
        const prom_layer &l = layers[i];
        if (l.cin < 1 || l.cin > 4096 || l.cout < 1 || l.cout > 4096) return false;
        if (i > 0 && l.cin != layers[i - 1].cout) return false;
        if (l.in_stride != 1 && l.in_stride != 2) return false;
        if (h % l.in_stride || w % l.in_stride) return false;
        // the block's input (the previous layer's input) has this layer's output shape
        if (l.add_block_input &&
            (i < 1 || l.in_stride != 1 || layers[i - 1].in_stride != 1 || l.cout != layers[i - 1].cin))
            return false;
        RowMap mp;
        mp.stride = l.in_stride; mp.hin = h; mp.win = w;
        h /= l.in_stride; w /= l.in_stride;
        mp.ho = h; mp.wo = w;
        if (l.dw_w) {                 // the depthwise convolution applies the stride itself
            if (l.cin & 3) return false;
            mp.stride = 1; mp.hin = h; mp.win = w;
        }
        s.map.push_back(mp);
        s.m.push_back((long long)batch * h * w);
        s.h.push_back(h); s.w.push_back(w);
    }
    return true;
}

// Workspace regions: a and b take the outputs of even and odd layers in turn; b also ends with
// room for the largest depthwise output (the input of the pointwise convolution behind it).
static void seq_regions(const prom_layer *layers, int n, const SeqShape &s, size_t &a, size_t &b,
                        size_t *dw_off = nullptr)
{
    a = b = 0;
    size_t c = 0;
    for (int i = 0; i < n; ++i) {
        if (i + 1 < n) {
            size_t bytes = round256((size_t)s.m[i] * layers[i].cout);
            if (i & 1) { if (bytes > b) b = bytes; }
            else { if (bytes > a) a = bytes; }
        }
        if (layers[i].dw_w) {
            size_t bytes = round256((size_t)s.m[i] * layers[i].cin);
            if (bytes > c) c = bytes;
        }
    }
    if (dw_off) *dw_off = a + b;
    b += c;
}

// ---- depth-first chains (chain.cuh) ---------------------------------------------------------
// A chain is a run of consecutive layers of a sequence that one launch of tc_chain_kernel takes
// tile by tile through all of them: same number of rows in every layer (only the first may
// subsample its input), channel counts that are multiples of 16, the clamp [0, 127], no
// depthwise convolution and no skip connection, and few enough tiles that a CTA interleaves
// at most chain::kMaxTasks of them.  Each layer of a chain writes to a buffer of its own in the
// workspace (a ping-pong pair would be overwritten by tiles that are layers ahead).
struct ChainPlan {
    int first = 0, last = 0;             // layers [first, last]
    int tm = 128, n_tasks = 0, grid = 0, box_r = 0;
    std::vector<TcPlan> prep;            // per layer: the plan whose image layout the kernel reads
    // kind 1: the run stays in shared memory (stack.cuh); `prep` is then empty
    int kind = 0;
    stack::Table st;                     // everything but pointers and tensor maps
    size_t smem = 0;
};

// Global scratch of one layer of a resident run: the int8 matrix, bias digits and constants that
// wide_prep_kernel writes, column tile after column tile.
struct StackScratch { size_t w8, wbias, consts, total; int n_ct, k_pad; };
static StackScratch stack_scratch(int cin, int cout)
{
    StackScratch z;
    z.n_ct = (cout + 127) / 128;
    z.k_pad = (cin + 127) / 128 * 128;
    z.w8 = (size_t)z.n_ct * 128 * z.k_pad;
    z.wbias = (size_t)z.n_ct * stack::kWbiasBytes;
    z.consts = round256((size_t)z.n_ct * stack::kConstBytes);
    z.total = z.w8 + z.wbias + z.consts;
    return z;
}

// The layers of a resident run alternate: P layers (the first and every second one after it; at
// most 384 output channels) and E layers (at most 384 input channels).
static bool stack_layer_ok(const prom_layer &l, bool is_p)
{
    if (l.dw_w || l.add_block_input || l.cin % 16 || l.cout % 16 || l.cin > 4096 || l.cout > 4096) return false;
    return is_p ? l.cout <= 128 * stack::kNarrowMax : l.cin <= 128 * stack::kNarrowMax;
}

// Roles, accumulator slots, shared-memory layout and rings of a resident run over the layers
// [c.first, c.last]; false when it does not fit.
static bool stack_fill(const prom_layer *layers, const DeviceInfo &d, ChainPlan &c)
{
    stack::Table &t = c.st;
    memset(&t, 0, sizeof(t));
    const int n = c.last - c.first + 1;
    if (n < 2 || n > stack::kMaxLayers) return false;
    int narrow = 1, ring_chunks = 0;
    for (int l = 0; l < n; ++l) {
        const prom_layer &pl = layers[c.first + l];
        stack::Layer &L = t.layer[l];
        L.cout = pl.cout;
        L.kc = (pl.cin + 127) / 128;
        L.ksteps = (pl.cin + 31) / 32;
        L.n_ct = (pl.cout + 127) / 128;
        L.act_min = pl.rq.act_min; L.act_max = pl.rq.act_max;
        L.streamed = (l & 1) ? 0 : 1;
        L.out_mode = l == n - 1 ? 2 : (L.streamed ? 0 : 1);
        if (L.streamed) {
            if (L.n_ct > stack::kNarrowMax) return false;
            L.ring_off = ring_chunks;
            ring_chunks += L.kc;
            if (L.out_mode == 0 && L.n_ct > narrow) narrow = L.n_ct;
        } else if (L.kc > stack::kNarrowMax) {
            return false;
        }
    }
    // accumulators: a P layer keeps all of its units' live, two of the four slots unless it has three
    // units; the E layer in front of it takes what is left
    for (int l = 0; l < n; ++l) {
        stack::Layer &L = t.layer[l];
        if (L.streamed) {
            L.nslots = L.n_ct == 3 ? 3 : 2;
            L.slot0 = stack::kAccs - L.nslots;
        } else {
            const bool tight = l + 1 < n && t.layer[l + 1].n_ct == 3;
            L.slot0 = 0;
            L.nslots = tight ? 1 : 2;
        }
    }
    t.n_layers = n;
    t.tm = c.tm; t.box_r = c.box_r; t.x3d = c.box_r > 0 ? 1 : 0;
    t.n_mtiles = c.n_tasks;
    t.chunks_per_tile = ring_chunks;
    t.ring = 3;
    const uint32_t const_bytes = stack::kAccs * stack::kSlotBytes;
    const uint32_t fixed = const_bytes + stack::kEpiWarps * stack::kSlabBytes + tc::kAConstBytes + 1024;
    const uint32_t act_bytes = (uint32_t)(narrow + t.ring) * stack::kChunkBytes;
    const long long room = (long long)d.smem_optin - 1024 - act_bytes - fixed;
    int stages = (int)(room / stack::kChunkBytes);
    if (stages > stack::kMaxStages) stages = stack::kMaxStages;
    stages &= ~1;                   // one half of the ring per issuing thread
    if (stages < 4) return false;
    t.stages = stages;
    t.off_nar = 0;
    t.off_ring = (uint32_t)narrow * stack::kChunkBytes;
    t.off_w = t.off_ring + (uint32_t)t.ring * stack::kChunkBytes;
    t.off_aconst = t.off_w + (uint32_t)stages * stack::kChunkBytes;
    t.off_const = t.off_aconst + tc::kAConstBytes;
    t.off_out = t.off_const + const_bytes;
    t.off_bars = t.off_out + stack::kEpiWarps * stack::kSlabBytes;
    c.smem = t.off_bars + 1024 + 1024;
    // one CTA per SM whatever the size: each allocates all of tensor memory
    if (c.smem < (size_t)d.smem_optin / 2 + 2048) c.smem = (size_t)d.smem_optin / 2 + 2048;
    return true;
}

static int chain_nt(int cout)
{
    if (cout % 16) return 0;
    if (cout <= chain::kNtMax) return cout;
    for (int nt = chain::kNtMax; nt >= 16; nt -= 16)
        if (cout % nt == 0) return nt;
    return 0;
}

static bool chain_layer_ok(const prom_layer &l)
{
    return !l.dw_w && !l.add_block_input && l.cin % 16 == 0 && l.cin >= 32 && l.cout % 16 == 0 &&
           l.rq.act_min == 0 && l.rq.act_max == 127 && chain_nt(l.cout) > 0;
}

static bool chain_prep_plan(long long m, int cin, int cout, const DeviceInfo &d, TcPlan &pl)
{
    const int nt = chain_nt(cout);
    const RowMap plain{1, 1, 1, 1, 1};
    return nt > 0 && tc_fill_plan(m, cin, cout, plain, d, 1, nt, cout / nt, 1, 0, pl, chain::kCwMax) &&
           pl.p.cw <= chain::kCwMax && pl.p.nt_pad <= chain::kNtMax &&
           (uint32_t)pl.p.nt_pad * 12u + 16u <= chain::kConstSlot;
}

static void find_chains(const prom_layer *layers, int n, const SeqShape &s, const DeviceInfo &d,
                        std::vector<ChainPlan> &out)
{
    out.clear();
    const int mode = g_seq_chain.load();
    if (!mode) return;
    int i = 0;
    while (mode == 2 && i < n) {
        // runs that stay in shared memory: P, E, P, E, ...
        if (!stack_layer_ok(layers[i], true) || s.m[i] <= 0 || s.m[i] + 256 >= (1ll << 31)) { ++i; continue; }
        ChainPlan c;
        c.kind = 1;
        c.first = i;
        const RowMap &mp = s.map[i];
        if (mp.stride != 1) {
            if (mp.wo > 128) { ++i; continue; }
            c.box_r = 128 / mp.wo;
            const long long lines = s.m[i] / mp.wo;
            if (c.box_r > lines) c.box_r = (int)lines;
            c.tm = c.box_r * mp.wo;
        }
        c.n_tasks = (int)((s.m[i] + c.tm - 1) / c.tm);
        int j = i + 1;
        while (j < n && j - i < stack::kMaxLayers && s.m[j] == s.m[i] && s.map[j].stride == 1 &&
               stack_layer_ok(layers[j], ((j - i) & 1) == 0))
            ++j;
        // the longest run that fits
        bool found = false;
        for (; j - i >= 2 && !found; --j) {
            // a skip connection into layer j reads the output of layer j - 2, which must exist
            if (j < n && layers[j].add_block_input) continue;
            c.last = j - 1;
            found = stack_fill(layers, d, c);
        }
        if (!found) { ++i; continue; }
        c.grid = c.n_tasks < d.sms ? c.n_tasks : d.sms;
        out.push_back(c);
        i = c.last + 1;
    }
    if (mode == 2) return;
    while (i < n) {
        if (!chain_layer_ok(layers[i]) || s.m[i] <= 0) { ++i; continue; }
        ChainPlan c;
        c.first = i;
        const RowMap &mp = s.map[i];
        if (mp.stride != 1) {
            if (mp.wo > 128) { ++i; continue; }
            c.box_r = 128 / mp.wo;
            const long long lines = s.m[i] / mp.wo;
            if (c.box_r > lines) c.box_r = (int)lines;
            c.tm = c.box_r * mp.wo;
        }
        const long long tasks = (s.m[i] + c.tm - 1) / c.tm;
        if (tasks > (long long)chain::kMaxTasks * 2 * d.sms || s.m[i] + 256 >= (1ll << 31)) { ++i; continue; }
        c.n_tasks = (int)tasks;
        int j = i;
        for (; j < n && j - i < chain::kMaxLayers; ++j) {
            if (!chain_layer_ok(layers[j]) || s.m[j] != s.m[i] || (j > i && s.map[j].stride != 1)) break;
            TcPlan pl;
            if (!chain_prep_plan(s.m[j], layers[j].cin, layers[j].cout, d, pl)) break;
            c.prep.push_back(pl);
        }
        if (j - i < 2) { ++i; continue; }
        c.last = j - 1;
        c.grid = c.n_tasks < 2 * d.sms ? c.n_tasks : 2 * d.sms;
        out.push_back(c);
        i = j;
    }
}

static bool make_x_map(CUtensorMap *map, const int8_t *x, int cin, long long rows, int cw, const RowMap *strided,
                       int box_r)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const CUtensorMapSwizzle sw = cw == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                  : (cw == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    cuuint32_t es[3] = {1, 1, 1};
    if (!strided) {
        cuuint64_t dims[2] = {(cuuint64_t)cin, (cuuint64_t)rows};
        cuuint64_t strides[1] = {(cuuint64_t)cin};
        cuuint32_t box[2] = {(cuuint32_t)cw, 128};
        return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(x), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    // [channel][wo, step stride*cin][batch*ho, step stride*win*cin]
    const RowMap &mp = *strided;
    cuuint64_t dims[3] = {(cuuint64_t)cin, (cuuint64_t)mp.wo, (cuuint64_t)(rows / mp.wo)};
    cuuint64_t strides[2] = {(cuuint64_t)mp.stride * cin, (cuuint64_t)mp.stride * mp.win * cin};
    cuuint32_t box[3] = {(cuuint32_t)cw, (cuuint32_t)mp.wo, (cuuint32_t)box_r};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t *>(x), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static bool make_y_map(CUtensorMap *map, int8_t *y, int nf, long long rows, int nt)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)nf, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)nf};
    cuuint32_t box[2] = {(cuuint32_t)nt, 32};
    cuuint32_t es[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, y, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- depthwise kernels: which one, for the layers and for the rule on blocks ----------------------
// 0: the library's choice, 1: CUDA cores only, 2: tensor cores or PROM_ERR_UNSUPPORTED
static std::atomic<int> g_dw_variant{0};
// Outputs from which the tensor-core kernel (dwtc.cuh) is the better one: a call of it costs about 6 us whatever its
// size (tensor memory and weight blocks to set up, one CTA of 190 KB per SM, so that little of this
// overlaps the kernel in front) against 3 us, and then 0.4 us per million outputs against 1.0 (stride 1)
// and 0.8 against 1.8 (stride 2).  Measured alone the lines cross at 3.3 to 5.6 million, inside the
// network's body at 3 to 6 million.
constexpr long long kDwTcOutputs = 4ll << 20;

// ---- whole blocks of a sequence in one launch (block.cuh) ------------------------------------------
// g_block_mode: 0: the library's choice, 1: never, 2: wherever a block qualifies; with a band height and a number of
// CTAs per cluster for tests (0: the planner's)
static std::atomic<int> g_block_mode{0}, g_block_rows{0}, g_block_split{0};

struct BlockPlan {
    block::Params p;
    int grid = 0;
    size_t smem = 0, image_bytes = 0;
    double est_us = 0;                      // of the geometry: what block_plan ranks by
    double block_us = 0, layers_us = 0;     // block_estimate
};

// Clusters of block_kernel that can be counted on to run at once.  A GPU holds 74, 45, 33, 26, 22, 15 and 15 of them
// (a cluster lies within one of its processing clusters), but behind a kernel that leaves its SMs one by one they do not
// pack like that: 45 clusters of three, 88 -> 528 -> 88 on 45 images of 12 x 12, took 16 us or 29 inside a sequence.
static int block_resident(int csize, const DeviceInfo &d)
{
    static const int b200[block::kMaxCluster + 1] = {0, 148, 66, 40, 29, 23, 19, 13, 13};
    const int n = d.sms >= 148 ? b200[csize] : d.sms / csize * 9 / 10;
    return n > 0 ? n : 1;
}

// The geometry of one candidate: `rows` output rows per band, `ipi` images per item, `per_cta` slices per CTA.
static bool block_fill(int c0, int ce, int co, int batch, int h, int w, int stride, int rows, int ipi, int per_cta,
                       const DeviceInfo &d, BlockPlan &pl)
{
    block::Params &p = pl.p;
    memset(&p, 0, sizeof(p));
    p.batch = batch; p.h = h; p.w = w; p.stride = stride;
    p.ho = (h - 1) / stride + 1; p.wo = (w - 1) / stride + 1;
    p.c0 = c0; p.co = co; p.npad = round_up(co, 16);
    p.rows = rows; p.rin = stride == 1 ? rows + 2 : 2 * rows + 1;
    p.bands = (p.ho + rows - 1) / rows; p.ipi = ipi;
    if (ipi > 1 && p.bands != 1) return false;
    const long long items = (long long)((batch + ipi - 1) / ipi) * p.bands;
    if (items >= (1 << 30) || (long long)batch * h >= (1ll << 31) || p.rin > 255 || ipi > 255) return false;
    p.items = (int)items;
    p.pitch = p.wo + 1;
    p.qlen = stride == 1 ? p.rin * p.pitch : (rows + 1) * p.pitch;
    const long long last = (long long)(ipi - 1) * p.qlen + (rows - 1) * p.pitch + p.wo;       // outputs in the buffer's order
    const long long pixels = (long long)ipi * p.rin * w;
    if (last > 128 * 16 || pixels > 128 * 24) return false;
    p.t1 = (int)((pixels + 127) / 128); p.t2 = (int)((last + 127) / 128);
    p.ks = (c0 + 31) / 32;
    p.slices = (ce + block::kSlice - 1) / block::kSlice;
    p.per_cta = per_cta;
    p.csize = (p.slices + per_cta - 1) / per_cta;
    if (p.csize > block::kMaxCluster) return false;
    // pixel buffer: what the last output block's taps reach, and where the expanded pixels go
    int reach = stride == 1 ? 128 * p.t2 + 2 * p.pitch + 3 : 128 * p.t2 + p.pitch + 2;
    const int held = ipi * p.qlen + 2;
    p.plane = round_up(reach > held ? reach : held, 8);
    const int len = stride == 1 ? p.plane : 4 * p.plane;
    if (len > 65535) return false;
    p.e_bytes = (uint32_t)round_up(len * block::kSlice, 1024);
    p.last_half = (ce - 1) % block::kSlice < block::kHalf;
    for (int dy = 0; dy < 3; ++dy)
        for (int dx = 0; dx < 3; ++dx)
            p.tap[3 * dy + dx] = (stride == 1 ? dy * p.pitch + dx
                                              : ((dy & 1) * 2 + (dx & 1)) * p.plane + (dy >> 1) * p.pitch + (dx >> 1)) *
                                 block::kSlice / 16;
    p.px = (c0 & 15) ? c0 / 8 : c0 / 16;
    p.px_magic = (uint32_t)(((1ull << 32) + p.px - 1) / p.px);
    if (pixels * p.px >= (1 << 20) || (long long)ipi * h * w * c0 >= (1ll << 31)) return false;
    p.x_bytes = (uint32_t)(p.t1 * p.ks) * block::kStepBytes;
    p.slice_bytes = block::slice_bytes(p.ks, p.npad);
    pl.image_bytes = (size_t)p.slices * p.slice_bytes;
    p.rpc = (ipi * rows * p.wo + p.csize - 1) / p.csize;
    p.xpitch = co + 4;
    auto magic = [](int v) { return v > 1 ? (uint32_t)(((1ull << 32) + v - 1) / v) : 0u; };
    p.per_img_magic = magic(p.rin * w); p.w_magic = magic(w); p.qlen_magic = magic(p.qlen); p.pitch_magic = magic(p.pitch);
    // tensor memory
    const int d3 = p.t2 * p.npad, cols = 512;
    p.n1 = 4; p.n2 = 4;
    p.chunks = p.t2 * ((co + 31) / 32);
    while (block::kSlice * (p.n1 + p.n2) + d3 > cols && p.n1 + p.n2 > 2) { if (p.n2 >= p.n1) p.n2 /= 2; else p.n1 /= 2; }
    if (block::kSlice * (p.n1 + p.n2) + d3 > cols) return false;
    p.d2_col = block::kSlice * p.n1; p.d3_col = p.d2_col + block::kSlice * p.n2;
    p.tmem_cols = cols;
    while (p.tmem_cols > 32 && p.d3_col + d3 <= p.tmem_cols / 2) p.tmem_cols /= 2;
    // shared memory: rings as deep as fit
    auto layout = [&](int ne, int ns, int np, int nx) {
        p.ne = ne; p.ns = ns; p.np = np; p.nx = nx;
        uint32_t o = (uint32_t)nx * p.x_bytes;
        p.off_e = o; o += (uint32_t)ne * p.e_bytes;
        p.off_p = o; o += (uint32_t)np * block::kUnitBytes;
        p.off_w = (o + 1023u) & ~1023u; o = p.off_w + (uint32_t)ns * p.slice_bytes;
        const uint32_t exch = (uint32_t)(p.csize > 1 ? p.csize * p.rpc * p.xpitch * 4 : 0);
        if (o < exch) o = exch;
        p.off_aconst = (o + 1023u) & ~1023u; o = p.off_aconst + tc::kAConstBytes;
        p.off_etab = o; o += 512u * (uint32_t)p.t1;
        p.off_otab = o; o += 512u * (uint32_t)p.t2;
        p.off_pc = o; o += 16u * (uint32_t)p.npad;
        p.off_bars = (o + 15u) & ~15u; o = p.off_bars + block::kBarBytes + 32u;
        return (size_t)o + 1024;
    };
    const bool one_item = p.csize > 1;
    static const int rings[][4] = {{4, 5, 4, 2}, {4, 4, 4, 2}, {4, 4, 4, 1}, {4, 4, 2, 1}, {2, 4, 4, 2}, {2, 3, 4, 2}, {2, 3, 2, 2}, {2, 3, 4, 1}, {2, 3, 2, 1}, {2, 2, 2, 1}};
    bool fits = false;
    for (const auto &r : rings) {
        int ns = r[1], nx = one_item ? 1 : r[3], ne = r[0], np = r[2];
        if (p.items <= d.sms) nx = 1;          // one item per CTA
        if (one_item && ns > per_cta) ns = per_cta;
        if (one_item) while (ne > per_cta) ne /= 2;
        p.ahead = ne > 1 ? ne - 1 : 1;
        pl.smem = layout(ne, ns, np, nx);
        if ((fits = pl.smem <= (size_t)d.smem_optin)) break;
    }
    if (!fits) return false;
    // a cluster takes one item; single CTAs stay and take one after the other
    const long long room = d.sms;
    p.clusters = p.csize > 1 ? p.items : (int)(p.items < room ? p.items : room);
    pl.grid = p.clusters * p.csize;
    // Time model, in cycles, fitted to 18 thousand timings (3297 shapes of the networks in several geometries; standard
    // error 8 %, the chosen geometry within 1 % of the best timed one on average).  What counts are the tensor pipe's
    // reads of shared memory (an MMA of 32 columns reads 5 KB, beside the epilogue's traffic), slices that are not asked
    // for early enough, what surrounds an item, and the rounds of resident clusters.
    const double tensor = 1.88 * (p.t1 * 48.0 * (p.ks + 1) + p.t2 * (800.0 + (p.npad > 80 ? p.npad : 80))) *
                          (p.slices - 0.5 * p.last_half) / p.slices;
    const int mine = p.csize > 1 ? 1 : (p.items + p.clusters - 1) / p.clusters;
    const int resident = block_resident(p.csize, d);
    const int waves = p.csize > 1 ? (p.items + resident - 1) / resident : 1;
    const bool late = p.ns < p.ahead + 2 && p.per_cta * mine > p.ns;
    const double slice = tensor + 680.0 / p.ahead + (late ? 540.0 + p.slice_bytes / 640.0 : 0.0);
    const double around = 4440.0 + tensor + (p.csize > 1 ? 7540.0 + 10.8 * p.t2 * p.npad : 0.0);
    const double item = 777.0 * p.t1 + (p.csize > 1 ? 0.0 : 4090.0 * ((p.chunks + block::kGroups - 1) / block::kGroups));
    pl.est_us = (8625.0 + waves * (around + (double)p.per_cta * mine * slice) + mine * item) / 1900.0;
    return true;
}

// Whether layers l[0], l[1] (rows of batch images of h x w pixels) are a block that block_kernel takes.
static bool block_layers_ok(const prom_layer *l)
{
    const prom_layer &e = l[0], &q = l[1];
    return !e.dw_w && e.in_stride == 1 && !e.add_block_input && q.dw_w && (e.cin & 7) == 0 && (e.cout & 7) == 0 &&
           (q.cout & 7) == 0 && q.cout <= 384 && e.cin <= 512 && e.cout >= 32;
}

// Whether the expanding layer and the depthwise convolution have the clamp that block_kernel's fast epilogues take.  With any
// other it computes by the 64-bit definition, the separate kernels mostly do not: with -128 in the expanding layer three blocks
// of 64 x 28 x 28, 32 -> 192 -> 32, took 125 us against 67, with an upper limit of 100 in the depthwise one 149 against 115;
// 32 x 14 x 14, 96 -> 576 -> 96, 93 against 55 and 100 against 57.
static bool block_clamps_fast(const prom_layer *l)
{
    return l[0].rq.act_min == 0 && l[0].rq.act_max == 127 && l[1].dw_rq.act_min == 0 && l[1].dw_rq.act_max == 127;
}

// What a call of one block alone is expected to take, in one launch and in one per layer (us).  Fits to 4942 shapes, blocks of
// the networks and others, standard errors 6.3 and 7.0 %, no worse on a third that a fit has not seen.  The planners' own
// figures go into both: that of the geometry here, those of the two pointwise layers there.
static void block_estimate(const prom_layer *l, const DeviceInfo &d, BlockPlan &pl)
{
    const block::Params &p = pl.p;
    const int ce = l[0].cout;
    const int more = p.csize > 1 ? 0 : (p.items + p.clusters - 1) / p.clusters - 1;      // items after a CTA's first
    const double e0 = pl.est_us - 4.54, pieces = 0.128 * p.t1 * p.px, sums = 0.01 * p.t2 * p.npad;
    pl.block_us = 4.83 + 0.7275 * e0 + (0.243 + 2.49 * more) * pieces + 0.523 * p.per_cta +
                  (p.csize > 1 ? 1.937 * sums
                               : 0.475 * more * sums + 0.133 * p.t1 + 0.0112 * (p.co < 48 ? 0 : p.co - 48) + (p.stride == 2 ? 0.052 * e0 : 0.0));
    TcPlan e, q;
    const int use = kPlanPrepared | kPlanOdd;
    pl.layers_us = 1e9;                     // not on the tensor cores: several times slower
    if (!tc_shape_plan((long long)p.batch * p.h * p.w, p.c0, ce, RowMap{1, 1, 1, 1, 1}, d, e, use) ||
        !tc_shape_plan((long long)p.batch * p.ho * p.wo, ce, p.co, RowMap{1, 1, 1, 1, 1}, d, q, use))
        return;
    const double out = (double)p.batch * p.ho * p.wo * ce * 1e-6;
    const bool odd_e = (p.c0 & 15) != 0, odd_p = ((ce | p.co) & 15) != 0, tensor_taps = (ce & 15) == 0 && out * 1e6 >= (double)kDwTcOutputs;
    pl.layers_us = 2.35 + (odd_e ? 0.722 : 0.64) * e.est_us + (odd_p ? 1.727 + 1.013 * q.est_us : 1.439 * q.est_us) +
                   2.007 * (out < 2.0 ? out : 2.0) + (tensor_taps ? 2.58 + 0.3 * out : (odd_p ? 0.997 : 0.66) * out) +
                   0.04 * (e.p.groups + q.p.groups);
}

// Whether one launch is expected to beat one per layer beside other blocks; the layers' time (us) is a fit to the shapes that
// the geometry's model was fitted to (standard error 7 %).  Inside a sequence a block saves about 1.2 us more than calls of its
// own show, whose preparation is not shared; its own estimate is low where the project layer is wide (more sums to exchange
// and to requantise) and with stride 2.  Mostly blocks are planes of 10 to 60 thousand pixels, batch included: larger ones
// are bound by the requantiser and the taps either way, and units leave gaps.  123 bodies of the network (five widths,
// four sizes, batch 1 to 151) take 0.944 of the time of one launch per layer on average, 0.85 to 1.014.
static bool block_worth(const BlockPlan &pl, int ce)
{
    const block::Params &p = pl.p;
    const double in = (double)p.batch * p.h * p.w * ce * 1e-6, out = (double)p.batch * p.ho * p.wo * ce * 1e-6;
    const bool tensor_taps = (ce & 15) == 0 && out * 1e6 >= (double)kDwTcOutputs;
    const double weights = 1e-4 * p.c0 * ce;
    const double layers = 12.4 + 0.27 * in + 2.26 * (out < 2.0 ? out : 2.0) + (tensor_taps ? 1.7 + 0.35 * out : 0.45 * out) +
                          0.19 * weights + 1.5 * out * p.co / ce + (p.c0 & 15 ? 0.15 * in + 0.26 * weights : 0.0) +
                          (p.co & 15 ? 0.13 + 0.083 * out : 0.0);
    const int wide = p.co < 48 ? 0 : p.co - 48;
    return pl.est_us * (1.0 + 0.0011 * wide + (p.stride == 1 ? 0.0 : p.csize == 1 ? 0.12 : 0.03)) - 1.2 < 0.96 * layers;
}

// What a call's blocks have to gain together, by block_estimate.  A block beside others, or beside other layers, gains
// kBlockBeside more than one whose call is nothing else (launches follow one another closer, the kernels of different layers
// wait for their instructions, the operands take one launch: 1.8 to 2.5 us per block in 130 bodies of the network).  So calls of
// one block alone need 0.5 us, and the bodies keep theirs.  Of 3391 such calls 0.2 % are slower than one launch per layer by
// more than 3 %, from a captured graph 0.7 % (without this rule, over the shapes of the fit, 1.7 and 4.7 %, up to 1.45 times).
// A block that block_estimate finds slower by more than 1.3 us is left to its layers where these are long enough for its figure
// to be the better one: 120 -> 720 -> 120 on 6 x 6 in a body of 86 images (425 us with it, 422 without, one launch per layer 417).
constexpr double kBlockBeside = 2.4, kBlocksGain = 0.5;
static bool block_slow(const BlockPlan &pl) { return pl.layers_us > 21.0 && pl.block_us > pl.layers_us + 1.3; }

typedef std::array<int, 10> BlockKey;
static bool block_plan(const prom_layer *l, int batch, int h, int w, const DeviceInfo &d, BlockPlan &best)
{
    const int c0 = l[0].cin, ce = l[0].cout, co = l[1].cout, stride = l[1].in_stride;
    const int f_rows = g_block_rows.load(), f_split = g_block_split.load();
    const BlockKey key = {c0, ce, co, batch, h, w, stride, d.dev, f_rows, f_split};
    static std::mutex mu;
    static std::map<BlockKey, std::pair<bool, BlockPlan>> cache;
    {
        std::lock_guard<std::mutex> lk(mu);
        const auto it = cache.find(key);
        if (it != cache.end()) {
            if (it->second.first) best = it->second.second;
            return it->second.first;
        }
    }
    // (not under the lock: other threads' known shapes need not wait for it)
    bool found = false;
    BlockPlan top;
    const int ho = (h - 1) / stride + 1, slices = (ce + block::kSlice - 1) / block::kSlice;
    for (int bands = 1; bands <= ho; ++bands) {
        const int rows = (ho + bands - 1) / bands;
        if (bands > 1 && rows == (ho + bands - 2) / (bands - 1)) continue;
        if (f_rows > 0 && rows != (f_rows < ho ? f_rows : ho)) continue;
        for (int ipi = 1; ipi <= (bands == 1 ? 8 : 1) && ipi <= batch; ++ipi)
            for (int c = 1; c <= block::kMaxCluster && c <= slices; ++c) {
                const int per = (slices + c - 1) / c;
                if ((slices + per - 1) / per != c) continue;
                if (f_split > 0 && c != f_split) continue;
                BlockPlan pl;
                if (!block_fill(c0, ce, co, batch, h, w, stride, rows, ipi, per, d, pl)) continue;
                if (!found || pl.est_us < top.est_us) { top = pl; found = true; }
            }
    }
    if (found) {
        block_estimate(l, d, top);
        best = top;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (cache.size() > 4096) cache.clear();
    cache.emplace(key, std::make_pair(found, top));
    return found;
}

static prom_status launch_block(BlockPlan &pl, const int8_t *x, int8_t *y, const int8_t *res, const uint8_t *image,
                                const prom_layer *l, int pdl, cudaStream_t st)
{
    block::Params &p = pl.p;
    p.x = x; p.y = y; p.res = res; p.image = image;
    p.bias = l[1].rq.bias; p.mult = l[1].rq.mult; p.shift = l[1].rq.shift;
    p.lo_e = l[0].rq.act_min; p.hi_e = l[0].rq.act_max;
    p.lo_d = l[1].dw_rq.act_min; p.hi_d = l[1].dw_rq.act_max;
    p.lo_p = l[1].rq.act_min; p.hi_p = l[1].rq.act_max;
    p.pdl = pdl;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    fill_launch_cfg(cfg, attr, pl.grid, block::kThreads, pl.smem, st, true);
    if (p.csize > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)p.csize;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, block::block_kernel, p);
    ++g_launches;
    return cuda_status(e);
}

// Where everything of a sequence sits in the caller's workspace.
struct SeqLayout {
    size_t ra = 0, rb = 0, dw_off = 0;     // the two ping-pong regions (b ends with the depthwise buffer)
    std::vector<size_t> img_off;           // per layer: prepared image of a one-launch layer, or -1
    size_t img_total = 0;
    std::vector<ChainPlan> chains;
    std::vector<int> chain_of;             // per layer: its chain, or -1
    std::vector<size_t> cimg_off, cbuf_off;   // per chain layer: images, output buffer
    size_t cimg_total = 0, cbuf_total = 0;
    std::vector<BlockPlan> blocks;         // layers taken two at a time by one launch
    std::vector<int> block_of;             // per layer: its block, or -1
    std::vector<size_t> bimg_off;          // per block: its slices' operands
    size_t bimg_total = 0;
    std::vector<char> region;              // per layer: the region its output goes to
    size_t plain_base = 0;                 // regions of one launch per layer (what a workspace must hold at least)
    size_t base() const { return ra + rb; }
    size_t with_images() const { return round256(base()) + img_total; }
    size_t with_blocks() const { return round256(with_images()) + bimg_total; }
    size_t with_chains() const { return round256(with_images()) + cimg_total + cbuf_total; }
};

// The blocks of a sequence: an expanding pointwise layer and, behind it, a layer with a depthwise convolution.
// What lies between them is not written, so the two regions take the outputs of what is left in turn.
static void find_blocks(const prom_layer *layers, int n, const SeqShape &s, const DeviceInfo &d, SeqLayout &L)
{
    const int mode = g_block_mode.load();
    if (mode == 1 || g_dw_variant.load() != 0) return;
    double gain = 0.0;
    for (int i = 0; i + 1 < n; ++i) {
        if (L.block_of[i] >= 0 || !block_layers_ok(layers + i) || s.m[i + 1] <= 0) continue;
        // a skip connection into layer i + 2 reads the expanded tensor, which must exist
        if (i + 2 < n && layers[i + 2].add_block_input) continue;
        BlockPlan pl;
        const int batch = (int)(s.m[i] / ((long long)s.h[i] * s.w[i]));
        if (!block_plan(layers + i, batch, s.h[i], s.w[i], d, pl)) continue;
        if (mode == 0 && !(block_clamps_fast(layers + i) && block_worth(pl, layers[i].cout) && !block_slow(pl))) continue;
        gain += pl.layers_us - pl.block_us + kBlockBeside;
        L.block_of[i] = L.block_of[i + 1] = (int)L.blocks.size();
        L.blocks.push_back(pl);
        L.bimg_off.push_back(L.bimg_total);
        L.bimg_total += round256(pl.image_bytes);
    }
    if (n == 2 * (int)L.blocks.size()) gain -= kBlockBeside;       // nothing else in the call
    if (mode == 0 && gain < kBlocksGain) {
        L.blocks.clear(); L.bimg_off.clear(); L.bimg_total = 0;
        L.block_of.assign(n, -1);
    }
    if (L.blocks.empty()) return;
    size_t r[2] = {0, 0}, c = 0;
    int side = 1;
    for (int i = 0; i < n; ++i) {
        const bool in_block = L.block_of[i] >= 0;
        if (in_block && i + 1 < n && L.block_of[i + 1] == L.block_of[i]) continue;         // has no output
        side ^= 1;
        L.region[i] = (char)side;
        const size_t bytes = round256((size_t)s.m[i] * layers[i].cout);
        if (i + 1 < n && bytes > r[side]) r[side] = bytes;
        if (layers[i].dw_w && !in_block) {
            const size_t b = round256((size_t)s.m[i] * layers[i].cin);
            if (b > c) c = b;
        }
    }
    L.ra = r[0]; L.rb = r[1] + c; L.dw_off = r[0] + r[1];
}

static void seq_layout(const prom_layer *layers, int n, const SeqShape &s, const DeviceInfo &d, bool want_tc,
                       SeqLayout &L, bool allow_chains = true, bool allow_blocks = true)
{
    seq_regions(layers, n, s, L.ra, L.rb, &L.dw_off);
    L.plain_base = L.base();
    L.chain_of.assign(n, -1);
    L.block_of.assign(n, -1);
    L.region.assign(n, 0);
    for (int i = 0; i < n; ++i) L.region[i] = (char)(i & 1);
    L.img_off.assign(n, (size_t)-1);
    L.cimg_off.assign(n, 0);
    L.cbuf_off.assign(n, 0);
    if (!want_tc || !d.ok) return;
    if (allow_chains) find_chains(layers, n, s, d, L.chains);
    if (allow_blocks && L.chains.empty()) find_blocks(layers, n, s, d, L);
    for (size_t c = 0; c < L.chains.size(); ++c)
        for (int i = L.chains[c].first; i <= L.chains[c].last; ++i) L.chain_of[i] = (int)c;
    for (int i = 0; i < n; ++i) {
        if (L.block_of[i] >= 0) continue;
        if (L.chain_of[i] >= 0) {
            const ChainPlan &c = L.chains[L.chain_of[i]];
            L.cimg_off[i] = L.cimg_total;
            if (c.kind == 1) {
                L.cimg_total += round256(stack_scratch(layers[i].cin, layers[i].cout).total);
                continue;
            }
            const tc::Params &p = c.prep[i - c.first].p;
            L.cimg_total += round256((size_t)p.groups * p.image_stride);
            continue;
        }
        TcPlan pl;
        if (tc_shape_plan(s.m[i], layers[i].cin, layers[i].cout, s.map[i], d, pl, kPlanPrepared | kPlanOdd)) {
            L.img_off[i] = L.img_total;
            L.img_total += round256((size_t)pl.p.groups * pl.p.image_stride);
        }
    }
    for (int i = 0; i < n; ++i)
        if (L.chain_of[i] >= 0 && i + 1 < n) {
            // (the inner layers of a resident run have no output tensor)
            const ChainPlan &c = L.chains[L.chain_of[i]];
            if (c.kind == 1 && i != c.last) continue;
            L.cbuf_off[i] = L.cimg_total + L.cbuf_total;
            L.cbuf_total += round256((size_t)s.m[i] * layers[i].cout);
        }
}

// ---- depthwise 3x3 on the tensor cores (dwtc.cuh) ---------------------------------------------
template <int STRIDE>
static prom_status launch_dw_tc(const int8_t *x, int batch, int h, int w, int c, const int8_t *wt,
                                const prom_requant *rq, int8_t *y, const DeviceInfo &d, cudaStream_t st, int pdl)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return PROM_ERR_UNSUPPORTED;
    dwtc::Params p;
    memset(&p, 0, sizeof(p));
    p.batch = batch; p.h = h; p.w = w; p.c = c;
    p.ho = (h - 1) / STRIDE + 1; p.wo = (w - 1) / STRIDE + 1;
    p.segs = (p.wo + 7) / 8;
    const long long groups = (long long)batch * p.segs;
    if (groups >= (1ll << 30) || h >= (1 << 30) || w >= (1 << 30)) return PROM_ERR_UNSUPPORTED;
    p.groups = (int)groups;
    p.blocks = (c + dwtc::kBlock - 1) / dwtc::kBlock;
    p.rows = (groups + dwtc::kGroups - 1) / dwtc::kGroups * p.ho;
    p.wt = wt; p.bias = rq->bias; p.mult = rq->mult; p.shift = rq->shift; p.lo = rq->act_min; p.hi = rq->act_max;
    p.y = y; p.pdl = pdl;
    if (p.blocks > d.sms) return PROM_ERR_UNSUPPORTED;
    // equal contiguous shares of the output rows; a share of a few rows would load mostly halo
    const long long workers = d.sms / p.blocks;
    long long per = (p.rows + workers - 1) / workers;
    const int least = STRIDE == 1 ? 6 : 3;
    if (per < least) per = least;
    if (per >= (1ll << 31)) return PROM_ERR_UNSUPPORTED;
    p.per_worker = (int)per;
    const int grid = (int)((p.rows + per - 1) / per) * p.blocks;
    // {channel, column, row, image}; with stride 2 one map of the odd and one of the even columns
    auto map_of = [&](CUtensorMap *m, const int8_t *base, int cols, int step, int px) {
        cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)cols, (cuuint64_t)h, (cuuint64_t)batch};
        cuuint64_t strides[3] = {(cuuint64_t)step * c, (cuuint64_t)w * c, (cuuint64_t)h * w * c};
        cuuint32_t box[4] = {(cuuint32_t)dwtc::kBlock, (cuuint32_t)px, (cuuint32_t)dwtc::kBoxRows, 1};
        cuuint32_t es[4] = {1, 1, 1, 1};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<int8_t *>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap xmap, emap;
    if (STRIDE == 1) {
        if (!map_of(&xmap, x, w, 1, dwtc::kPx)) return PROM_ERR_UNSUPPORTED;
        emap = xmap;        // unused
    } else {
        if (w < 2 || !map_of(&xmap, x + c, w / 2, 2, dwtc::kPx) || !map_of(&emap, x, (w + 1) / 2, 2, 8))
            return PROM_ERR_UNSUPPORTED;
    }
    const int smem = (int)dwtc::smem_bytes(STRIDE);
    if (raise_smem_limit(dwtc::dw3x3_tc_kernel<STRIDE>, smem) != cudaSuccess) return PROM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, grid, dwtc::kThreads, (size_t)smem, st, pdl != 0);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, dwtc::dw3x3_tc_kernel<STRIDE>, xmap, emap, p);
    ++g_launches;
    return cuda_status(e);
}

// pdl: how the kernel is chained to the previous one of the stream (tc.cuh: kPdl*); it may always
// be chained to
static prom_status dw_conv3x3(const int8_t *x_dev, int batch, int h, int w, int c, int stride,
                              const int8_t *w_dev, const prom_requant *rq, int8_t *y_dev, void *cuda_stream,
                              int pdl)
{
    if (batch < 0 || h < 1 || w < 1 || c < 1 || c > 4096 || (stride != 1 && stride != 2)) return PROM_ERR_SHAPE;
    if (c & 3) return PROM_ERR_UNSUPPORTED;
    if (!rq) return PROM_ERR_NULL;
    prom_status e = check_requant(rq);
    if (e != PROM_OK) return e;
    if (batch == 0) return PROM_OK;
    if (!x_dev || !w_dev || !y_dev) return PROM_ERR_NULL;
    if (!aligned16(x_dev) || !aligned16(y_dev)) return PROM_ERR_ALIGN;
    if (reinterpret_cast<const void *>(x_dev) == reinterpret_cast<const void *>(y_dev)) return PROM_ERR_ALIGN;
    const int ho = (h - 1) / stride + 1, wo = (w - 1) / stride + 1;
    if ((long long)batch * h * w * c >= (1ll << 40)) return PROM_ERR_SHAPE;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    // whole slices of 16 channels and enough work: TMA patches and tensor-core taps
    const int dw_variant = g_dw_variant.load();
    if (dw_variant != 1 && (c & 15) == 0 &&
        (dw_variant == 2 || (long long)batch * ho * wo * c >= kDwTcOutputs)) {
        cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
        const prom_status e = stride == 1 ? launch_dw_tc<1>(x_dev, batch, h, w, c, w_dev, rq, y_dev, d, st, pdl)
                                          : launch_dw_tc<2>(x_dev, batch, h, w, c, w_dev, rq, y_dev, d, st, pdl);
        if (e != PROM_ERR_UNSUPPORTED) return e;
    }
    if (dw_variant == 2) return PROM_ERR_UNSUPPORTED;
    // Units (dw3x3_kernel's ROWS x STRIP pixels of four channels, one per thread at a time): large ones read
    // fewer pixels twice, small ones give a small layer more threads and each of them less to do.
    int rows = stride == 1 ? 2 : 1, strip = 4;
    auto units_of = [&] { return (long long)batch * ((ho + rows - 1) / rows) * ((wo + strip - 1) / strip); };
    // (Inside a sequence the next layer waits for the slowest thread: body of the network at batch 9 and width
    // 0.75 285 -> 264 us, at batch 1 219 -> 200.  Calls of their own overlap, and there the work counts:
    // [9,28,28,144] 4.1 us against 5.7 with small units, [1,28,28,192] 3.5 against 2.8.)
    const bool small = units_of() * (c >> 2) < (pdl == tc::kPdlChain ? 300ll : 40ll) * d.sms;
    if (small) { rows = 1; strip = 2; }
    const long long units = units_of();
    if (units >= (1ll << 31)) return PROM_ERR_SHAPE;
    const long long total = units * (c >> 2);
    // a multiple of c / 4 threads, so that a thread keeps its channels: blocks in multiples of
    // (c / 4) / gcd(c / 4, threads per block)
    int step = c >> 2;
    for (int a = step, b = dw::kThreads; b;) { const int r = a % b; a = b; b = r; if (!b) step = (c >> 2) / a; }
    long long blocks = (total + dw::kThreads - 1) / dw::kThreads;
    const long long cap = (long long)d.sms * 16;
    if (blocks > cap) blocks = cap;
    blocks = (blocks + step - 1) / step * step;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, (int)blocks, dw::kThreads, 0, static_cast<cudaStream_t>(cuda_stream), pdl != 0);
    auto *kernel = stride == 1 ? (small ? dw::dw3x3_kernel<1, 1, 2> : dw::dw3x3_kernel<1, 2, 4>)
                               : (small ? dw::dw3x3_kernel<2, 1, 2> : dw::dw3x3_kernel<2, 1, 4>);
    const cudaError_t le = cudaLaunchKernelEx(&cfg, kernel, x_dev, batch, h, w, c, ho, wo, w_dev, rq->bias, rq->mult,
                                              rq->shift, rq->act_min, rq->act_max, y_dev, pdl);
    ++g_launches;
    return cuda_status(le);
}

// One launch of tc_chain_kernel for layers [c.first, c.last]; conv[] holds every layer's pointers.
static prom_status launch_chain(const prom_layer *layers, const SeqShape &s, const ChainPlan &c,
                                const std::vector<Conv> &conv, uint8_t *const *images, bool pdl, bool pdl_next,
                                cudaStream_t st)
{
    chain::Table t;
    memset(&t, 0, sizeof(t));
    t.m_rows = s.m[c.first];
    t.n_layers = c.last - c.first + 1;
    t.n_tasks = c.n_tasks;
    t.tm = c.tm;
    t.pdl = pdl ? 1 : 0;
    t.pdl_next = pdl_next ? 1 : 0;
    for (int i = c.first; i <= c.last; ++i) {
        chain::Layer &L = t.layer[i - c.first];
        const tc::Params &p = c.prep[i - c.first].p;
        const bool strided = i == c.first && s.map[i].stride != 1;
        if (!make_x_map(&L.xmap, conv[i].x, layers[i].cin, s.m[i], p.cw, strided ? &s.map[i] : nullptr, c.box_r))
            return PROM_ERR_CUDA;
        L.store_2d = p.n_sub > 1 ? 1 : 0;
        if (L.store_2d) {
            if (!make_y_map(&L.ymap, conv[i].y, layers[i].cout, s.m[i], p.nt)) return PROM_ERR_CUDA;
        } else {
            L.ymap = L.xmap;       // unused
        }
        L.image = images[i];
        L.y = conv[i].y;
        L.image_stride = p.image_stride;
        L.wbias_off = p.off_wbias - p.off_w;
        L.const_off = p.off_mult - p.off_w;
        L.const_bytes = (uint32_t)p.nt_pad * 12u + 16u;
        L.a_tx = strided ? (uint32_t)(p.cw * s.map[i].wo * c.box_r) : 128u * (uint32_t)p.cw;
        L.n = layers[i].cout;
        L.cw = p.cw; L.kc = p.kc; L.ksteps_last = p.ksteps_last;
        L.nt = p.nt; L.nt_pad = p.nt_pad; L.n_sub = p.n_sub;
        L.x3d = strided ? 1 : 0;
        L.box_r = c.box_r;
        L.act_min = layers[i].rq.act_min; L.act_max = layers[i].rq.act_max;
    }
    if (raise_smem_limit(chain::tc_chain_kernel, (int)chain::kSmemBytes) != cudaSuccess) return PROM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)c.grid);
    cfg.blockDim = dim3(chain::kThreads);
    cfg.dynamicSmemBytes = chain::kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (pdl) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, chain::tc_chain_kernel, t);
    ++g_launches;
    return cuda_status(e);
}

// One launch of stack_kernel for the layers [c.first, c.last] of a resident run.
static prom_status launch_stack(const prom_layer *layers, const SeqShape &s, const ChainPlan &c,
                                const std::vector<Conv> &conv, uint8_t *const *scratch, const DeviceInfo &d,
                                bool pdl, bool pdl_next, cudaStream_t st)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return PROM_ERR_CUDA;
    stack::Table t = c.st;
    t.m = s.m[c.first];
    t.pdl = pdl ? 1 : 0;
    t.pdl_next = pdl_next ? 1 : 0;
    t.y = conv[c.last].y;
    const bool strided = s.map[c.first].stride != 1;
    if (!make_x_map(&t.xmap, conv[c.first].x, layers[c.first].cin, s.m[c.first], 128,
                    strided ? &s.map[c.first] : nullptr, c.box_r))
        return PROM_ERR_CUDA;
    if (!make_y_map(&t.ymap, conv[c.last].y, layers[c.last].cout, s.m[c.last], 32)) return PROM_ERR_CUDA;
    cuuint32_t es[2] = {1, 1};
    for (int i = c.first; i <= c.last; ++i) {
        stack::Layer &L = t.layer[i - c.first];
        const StackScratch z = stack_scratch(layers[i].cin, layers[i].cout);
        cuuint64_t dims[2] = {(cuuint64_t)z.k_pad, (cuuint64_t)z.n_ct * 128};
        cuuint64_t strides[1] = {(cuuint64_t)z.k_pad};
        cuuint32_t box[2] = {128, 128};
        if (enc(&L.wmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, scratch[i], dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PROM_ERR_CUDA;
        L.wbias = scratch[i] + z.w8;
        L.consts = scratch[i] + z.w8 + z.wbias;
    }
    if (raise_smem_limit(stack::stack_kernel, d.smem_optin) != cudaSuccess) return PROM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, c.grid, stack::kThreads, c.smem, st, pdl);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, stack::stack_kernel, t);
    ++g_launches;
    return cuda_status(e);
}

static bool seq_overlap(const int8_t *a, size_t na, const int8_t *b, size_t nb) { return a < b + nb && b < a + na; }

static prom_status run_seq(const prom_layer *layers, int n, const int8_t *x0, int batch, int h0,
                           int w0, void *ws, size_t ws_bytes, int8_t *y_out, prom_variant variant,
                           cudaStream_t st)
{
    SeqShape s;
    if (!seq_shapes(layers, n, batch, h0, w0, s)) return PROM_ERR_SHAPE;
    // validate everything before the first launch
    for (int i = 0; i < n; ++i) {
        if (!layers[i].w_packed) return PROM_ERR_NULL;
        if (layers[i].dw_w) {
            prom_status de = check_requant(&layers[i].dw_rq);
            if (de != PROM_OK) return de;
        }
        prom_status e = check_requant(&layers[i].rq);
        if (e != PROM_OK) return e;
        if (!aligned16(layers[i].w_packed)) return PROM_ERR_ALIGN;
        if (layers[i].add_block_input &&
            (variant == PROM_VARIANT_SMALLK || variant == PROM_VARIANT_ADDSUB))
            return PROM_ERR_UNSUPPORTED;
    }
    DeviceInfo d = device_info();
    const bool want_tc = variant == PROM_VARIANT_TC || variant == PROM_VARIANT_AUTO;
    SeqLayout lay;
    seq_layout(layers, n, s, d, want_tc, lay);
    if (lay.plain_base > 0) {
        if (!ws) return PROM_ERR_NULL;
        if (!aligned16(ws)) return PROM_ERR_ALIGN;
        if (ws_bytes < lay.plain_base) return PROM_ERR_WORKSPACE;
    }
    if (!d.ok) return PROM_ERR_CUDA;
    // A block reads rows of its input that other CTAs' outputs stand for, so the two may not overlap; and
    // its operands need room.  One launch per layer takes any workspace of the plain size.
    if (!lay.blocks.empty() && (ws_bytes < lay.with_blocks() ||
                                seq_overlap(x0, (size_t)batch * h0 * w0 * layers[0].cin, y_out, (size_t)s.m[n - 1] * layers[n - 1].cout))) {
        lay = SeqLayout();
        seq_layout(layers, n, s, d, want_tc, lay, true, false);
    }
    int8_t *reg[2] = {static_cast<int8_t *>(ws), static_cast<int8_t *>(ws) + lay.ra};
    int8_t *dw_buf = static_cast<int8_t *>(ws) + lay.dw_off;      // depthwise outputs

    // The images and the chains are optimisations: a workspace without room for them still works.
    uint8_t *img_base = nullptr, *chain_base = nullptr;
    if (ws && lay.img_total + lay.cimg_total > 0 && ws_bytes >= lay.with_images())
        img_base = static_cast<uint8_t *>(ws) + round256(lay.base());
    if (ws && !lay.chains.empty() && ws_bytes >= lay.with_chains())
        chain_base = static_cast<uint8_t *>(ws) + round256(lay.with_images());
    if (!chain_base && !lay.chains.empty()) {
        // no room: plan again without chains (their layers then want one-launch images)
        lay = SeqLayout();
        seq_layout(layers, n, s, d, want_tc, lay, false, false);
        img_base = nullptr;
        if (ws && lay.img_total > 0 && ws_bytes >= lay.with_images())
            img_base = static_cast<uint8_t *>(ws) + round256(lay.base());
    }

    // plan: which layers run on the tensor cores, and where their prepared operands go
    std::vector<Conv> conv(n);
    std::vector<TcPlan> plan(n);
    std::vector<char> is_tc(n, 0);
    std::vector<uint8_t *> chain_img(n, nullptr);
    std::vector<const int8_t *> input(n, nullptr);
    uint8_t *block_base = lay.blocks.empty() ? nullptr : static_cast<uint8_t *>(ws) + round256(lay.with_images());
    const int8_t *cur = x0;
    long long in_rows = (long long)batch * h0 * w0;
    for (int i = 0; i < n; ++i) {
        Conv &c = conv[i];
        const bool chained = lay.chain_of[i] >= 0, in_block = lay.block_of[i] >= 0;
        input[i] = cur;
        // behind a depthwise convolution the pointwise layer reads that convolution's output
        c.x = layers[i].dw_w ? dw_buf : cur; c.m = s.m[i]; c.cin = layers[i].cin; c.cout = layers[i].cout;
        c.map = s.map[i]; c.in_rows = layers[i].dw_w ? s.m[i] : in_rows;
        c.w = layers[i].w_packed; c.rq = layers[i].rq;
        c.y = (i == n - 1) ? y_out
              : (chained ? reinterpret_cast<int8_t *>(chain_base + lay.cbuf_off[i]) : reg[(int)lay.region[i]]);
        c.st = st;
        // the first kernel waits before it reads anything (the operands prepared below included) and
        // before it releases its successor, so every later link finds weights and operands complete
        c.pdl = i > 0 || layers[i].dw_w ? tc::kPdlChain : tc::kPdlWait;
        c.pdl_next = true;
        // The input of layer i-1, often in the region that this layer's output goes to (a chain's layers write buffers
        // of their own).  It is always a tensor in memory: find_blocks and find_chains see to that.
        if (layers[i].add_block_input) c.res = input[i - 1];
        if (in_block) {
            // (what one launch per layer refuses stays refused)
            TcPlan tmp;
            if (variant == PROM_VARIANT_TC && !tc_shape_plan(c.m, c.cin, c.cout, c.map, d, tmp, kPlanPrepared)) return PROM_ERR_UNSUPPORTED;
            if (i + 1 < n && lay.block_of[i + 1] == lay.block_of[i]) continue;         // has no output: the next layer's input is this one's
        } else if (chained) {
            chain_img[i] = chain_base + lay.cimg_off[i];
        } else if (want_tc && c.m > 0 && tc_shape_plan(c.m, c.cin, c.cout, c.map, d, plan[i],
                                                               variant == PROM_VARIANT_AUTO ? kPlanPrepared | kPlanOdd : kPlanPrepared)) {
            is_tc[i] = 1;
            tc_bind(c, plan[i], img_base && lay.img_off[i] != (size_t)-1 ? img_base + lay.img_off[i] : nullptr);
        } else if (variant == PROM_VARIANT_TC && c.m > 0) {
            return PROM_ERR_UNSUPPORTED;
        }
        cur = c.y;
        in_rows = c.m;
    }
    if (want_tc && tc_set_attr(d) != PROM_OK) return PROM_ERR_CUDA;
    // tile order: opposite to that of the kernel that wrote the layer's input (a depthwise
    // convolution and the kernels off the tensor cores walk forwards)
    if (g_seq_snake.load()) {
        bool writer_rev = true;             // the first layer walks forwards
        for (int i = 0; i < n; ++i) {
            if (layers[i].dw_w) writer_rev = false;
            if (lay.block_of[i] >= 0) continue;
            const bool rev = is_tc[i] && lay.chain_of[i] < 0 && !writer_rev;
            if (is_tc[i]) plan[i].p.reverse = rev ? 1 : 0;
            writer_rev = rev;
        }
    }

    // one launch prepares the operands of every tensor-core layer (of a chain: one image per subtile)
    bool prepared = false;              // such a launch of this call is in front
    if (img_base || chain_base) {
        int i = 0;
        while (i < n) {
            tc::PrepTable t;
            memset(&t, 0, sizeof(t));
            size_t smem = 0;
            int ctas = 0;
            for (; i < n && t.n < tc::kMaxPrepLayers; ++i) {
                if (lay.chain_of[i] >= 0) {
                    const ChainPlan &c = lay.chains[lay.chain_of[i]];
                    if (c.kind == 1) continue;          // prepared by the batch below
                    TcPlan tmp = c.prep[i - c.first];
                    tc_bind(conv[i], tmp, chain_img[i]);
                    prep_add(t, tmp.p, ctas, smem);
                } else if (is_tc[i] && plan[i].p.image) {
                    prep_add(t, plan[i].p, ctas, smem);
                }
            }
            if (t.n == 0) break;
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[1];
            fill_launch_cfg(cfg, attr, ctas, tc::kPrepThreads, smem, st, true);
            const cudaError_t e = cudaLaunchKernelEx(&cfg, tc::tc_prep_kernel, t);
            prepared = true;
            ++g_launches;
            if (e != cudaSuccess) return PROM_ERR_CUDA;
        }
    }

    // ... one launch those of the blocks
    for (size_t k = 0; k < lay.blocks.size();) {
        block::PrepTable t;
        memset(&t, 0, sizeof(t));
        t.behind = prepared ? 1 : 0;
        prepared = true;
        int ctas = 0;
        for (; k < lay.blocks.size() && t.n < block::kMaxPrep; ++k) {
            int i = 0;
            while (lay.block_of[i] != (int)k) ++i;
            const block::Params &p = lay.blocks[k].p;
            const prom_layer &e = layers[i], &q = layers[i + 1];
            block::PrepBlock &b = t.b[t.n++];
            b.we = e.w_packed; b.wp = q.w_packed; b.wd = q.dw_w;
            b.bias_e = e.rq.bias; b.mult_e = e.rq.mult; b.shift_e = e.rq.shift;
            b.bias_d = q.dw_rq.bias; b.mult_d = q.dw_rq.mult; b.shift_d = q.dw_rq.shift;
            b.image = block_base + lay.bimg_off[k];
            b.c0 = e.cin; b.ce = e.cout; b.co = q.cout; b.npad = p.npad; b.ks = p.ks;
            b.lo_e = e.rq.act_min; b.hi_e = e.rq.act_max; b.lo_d = q.dw_rq.act_min; b.hi_d = q.dw_rq.act_max;
            b.first = ctas;
            ctas += p.slices;
        }
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        fill_launch_cfg(cfg, attr, ctas, block::kPrepThreads, 0, st, true);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, block::block_prep_kernel, t);
        ++g_launches;
        if (e != cudaSuccess) return cuda_status(e);
    }
    if (!lay.blocks.empty() && raise_smem_limit(block::block_kernel, d.smem_optin) != cudaSuccess) return PROM_ERR_CUDA;

    // ... and one launch the operands of the runs that stay in shared memory
    if (chain_base) {
        int i = 0;
        while (i < n) {
            wide::PrepBatch b;
            memset(&b, 0, sizeof(b));
            int ctas = 0;
            for (; i < n && b.n < wide::kMaxPrepLayers; ++i) {
                if (lay.chain_of[i] < 0 || lay.chains[lay.chain_of[i]].kind != 1) continue;
                const StackScratch z = stack_scratch(layers[i].cin, layers[i].cout);
                wide::PrepParams &pp = b.layer[b.n];
                pp.cin = layers[i].cin; pp.cout = layers[i].cout; pp.k_pad = z.k_pad; pp.w_packed = layers[i].w_packed;
                pp.bias = layers[i].rq.bias; pp.mult = layers[i].rq.mult; pp.shift = layers[i].rq.shift;
                pp.act_min = layers[i].rq.act_min; pp.act_max = layers[i].rq.act_max;
                pp.w8 = reinterpret_cast<int8_t *>(chain_img[i]);
                pp.wbias = chain_img[i] + z.w8;
                pp.consts = chain_img[i] + z.w8 + z.wbias;
                b.first[b.n] = ctas;
                ctas += z.n_ct;
                ++b.n;
            }
            if (b.n == 0) break;
            b.first[b.n] = ctas;
            wide::wide_prep_batch_kernel<<<ctas, 256, 0, st>>>(b);
            ++g_launches;
            if (cudaGetLastError() != cudaSuccess) return PROM_ERR_CUDA;
        }
    }

    for (int i = 0; i < n; ++i) {
        if (lay.chain_of[i] >= 0) {
            const ChainPlan &c = lay.chains[lay.chain_of[i]];
            prom_status e = c.kind == 1
                ? launch_stack(layers, s, c, conv, chain_img.data(), d, c.first > 0, c.last + 1 < n, st)
                : launch_chain(layers, s, c, conv, chain_img.data(), c.first > 0, c.last + 1 < n, st);
            if (e != PROM_OK) return e;
            i = c.last;
            continue;
        }
        if (lay.block_of[i] >= 0) {
            const int k = lay.block_of[i];
            const prom_status e = launch_block(lay.blocks[k], input[i], conv[i + 1].y, conv[i + 1].res, block_base + lay.bimg_off[k],
                                               layers + i, i > 0 ? tc::kPdlChain : tc::kPdlWait, st);
            if (e != PROM_OK) return e;
            ++i;
            continue;
        }
        if (layers[i].dw_w && s.m[i] > 0) {
            const int stride = layers[i].in_stride;
            const int8_t *src = input[i];
            // chained like the pointwise kernels: behind layer i-1's kernel (which releases its
            // dependents at entry) and in front of layer i's, which waits for it before its loads
            prom_status de = dw_conv3x3(src, batch, s.h[i] * stride, s.w[i] * stride, layers[i].cin, stride,
                                        layers[i].dw_w, &layers[i].dw_rq, dw_buf, st,
                                        i > 0 ? tc::kPdlChain : tc::kPdlWait);
            if (de != PROM_OK) return de;
        }
        prom_status e = is_tc[i] ? tc_launch_planned(conv[i], plan[i]) : run_conv(conv[i], variant);
        if (e != PROM_OK) return e;
    }
    return PROM_OK;
}

// ---- the add/sub variant on built-in scratch (no allocation anywhere) --------------------
// The index lists of the add/sub variant normally live in a buffer the library
// grows with cudaMalloc.  This copy of the scratch is part of the loaded module
// instead: PROM_STATIC_SCRATCH_BYTES of device memory on every GPU that loads
// the library, held until the process exits.  In host code the array's name is
// only a handle for the runtime, not a device address; the address a kernel can
// use comes from cudaGetSymbolAddress, asked once per device.
static __device__ __align__(256) uint8_t g_static_scratch[PROM_STATIC_SCRATCH_BYTES];

static uint8_t *static_scratch_address()
{
    static std::mutex mu;
    static std::unordered_map<int, uint8_t *> by_device;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    auto it = by_device.find(dev);
    if (it != by_device.end()) return it->second;
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return nullptr;
    by_device[dev] = static_cast<uint8_t *>(p);
    return static_cast<uint8_t *>(p);
}

// Clears the maxima of the dynamic layer (a kernel and not a memset, which would keep the passes behind it
// from being launched early).
__global__ void dyn_clear_kernel(float *__restrict__ gamma_y, int batch)
{
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < batch) gamma_y[b] = 0.0f;
}

}  // namespace prom

using namespace prom;

extern "C" {

size_t prom_packed_bytes(int cout, int cin)
{
    if (cout < 0 || cin < 0) return 0;
    return (size_t)cout * (size_t)((cin + 3) / 4);
}

prom_status prom_pack_ternary(const int8_t *w_dev, int cout, int cin, uint8_t *packed_dev,
                              size_t packed_bytes, void *cuda_stream)
{
    if (!w_dev || !packed_dev) return PROM_ERR_NULL;
    if (cout < 1 || cin < 1 || cout > 4096 || cin > 4096) return PROM_ERR_SHAPE;
    if (packed_bytes < prom_packed_bytes(cout, cin)) return PROM_ERR_WORKSPACE;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    unsigned int *bad = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void **>(&bad), g_pack_bad) != cudaSuccess)
        return PROM_ERR_CUDA;
    if (cudaMemsetAsync(bad, 0, sizeof(unsigned int), st) != cudaSuccess) return PROM_ERR_CUDA;
    long long total = (long long)cout * ((cin + 3) / 4);
    pack_ternary_kernel<<<grid_for(total, 256, d.sms), 256, 0, st>>>(w_dev, cout, cin, packed_dev,
                                                                     bad);
    ++g_launches;
    if (cudaGetLastError() != cudaSuccess) return PROM_ERR_CUDA;
    unsigned int host_bad = 0;
    if (cudaMemcpyAsync(&host_bad, bad, sizeof(host_bad), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return PROM_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return PROM_ERR_CUDA;
    return host_bad ? PROM_ERR_BAD_WEIGHT : PROM_OK;
}

prom_status prom_quantize_ternary(const float *w_dev, int cout, int cin, uint8_t *packed_dev,
                                  size_t packed_bytes, float *alpha_dev, void *cuda_stream)
{
    if (!w_dev || !packed_dev) return PROM_ERR_NULL;
    if (cout < 1 || cin < 1 || cout > 4096 || cin > 4096) return PROM_ERR_SHAPE;
    if (packed_bytes < prom_packed_bytes(cout, cin)) return PROM_ERR_WORKSPACE;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    const int want = (cout + quant::kWarps - 1) / quant::kWarps;        // a warp per row
    const int grid = want < d.sms * 16 ? want : d.sms * 16;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, grid, quant::kThreads, 0, static_cast<cudaStream_t>(cuda_stream), true);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, quant::quantize_ternary_kernel, w_dev, cout, cin, 1e-5, packed_dev,
                                             alpha_dev);
    ++g_launches;
    return cuda_status(e);
}

prom_status prom_quantize_ternary_batch(const prom_quantize_job *jobs, int n, void *cuda_stream)
{
    if (!jobs) return PROM_ERR_NULL;
    if (n < 0) return PROM_ERR_SHAPE;
    for (int i = 0; i < n; ++i) {
        const prom_quantize_job &j = jobs[i];
        if (!j.w_dev || !j.packed_dev) return PROM_ERR_NULL;
        if (j.cout < 1 || j.cin < 1 || j.cout > 4096 || j.cin > 4096) return PROM_ERR_SHAPE;
        if (j.packed_bytes < prom_packed_bytes(j.cout, j.cin)) return PROM_ERR_WORKSPACE;
    }
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    for (int base = 0; base < n; base += quant::kMaxJobs) {
        quant::Jobs t;
        memset(&t, 0, sizeof(t));
        t.n = n - base < quant::kMaxJobs ? n - base : quant::kMaxJobs;
        int rows = 0;
        for (int i = 0; i < t.n; ++i) {
            const prom_quantize_job &j = jobs[base + i];
            t.first_row[i] = rows;
            rows += j.cout;
            t.cin[i] = j.cin; t.w[i] = j.w_dev; t.packed[i] = j.packed_dev; t.alpha[i] = j.alpha_dev;
        }
        t.first_row[t.n] = rows;
        const int want = (rows + quant::kWarps - 1) / quant::kWarps;      // a warp per row
        const int grid = want < d.sms * 16 ? want : d.sms * 16;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        fill_launch_cfg(cfg, attr, grid, quant::kThreads, 0, static_cast<cudaStream_t>(cuda_stream), true);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, quant::quantize_ternary_batch_kernel, t, 1e-5);
        ++g_launches;
        if (e != cudaSuccess) return PROM_ERR_CUDA;
    }
    return PROM_OK;
}

prom_status prom_dw_conv3x3_i8(const int8_t *x_dev, int batch, int h, int w, int c, int stride,
                               const int8_t *w_dev, const prom_requant *rq, int8_t *y_dev,
                               void *cuda_stream)
{
    return dw_conv3x3(x_dev, batch, h, w, c, stride, w_dev, rq, y_dev, cuda_stream, tc::kPdlWait);
}

prom_status prom_pw_conv_i8_dyn(const int8_t *x_dev, int batch, int64_t rows_per_sample, int cin,
                                const uint8_t *w_packed_dev, int cout, const float *alpha_dev,
                                const float *gamma_x_dev, int8_t *q_dev, float *gamma_y_dev,
                                float *scale_y_dev, void *cuda_stream)
{
    if (batch < 0 || rows_per_sample < 1 || cin < 1 || cout < 1 || cin > 4096 || cout > 4096)
        return PROM_ERR_SHAPE;
    const long long m = (long long)batch * rows_per_sample;
    if (rows_per_sample >= (1ll << 31) || m >= (1ll << 31)) return PROM_ERR_SHAPE;
    if (batch == 0) return PROM_OK;
    if (!x_dev || !w_packed_dev || !alpha_dev || !gamma_x_dev || !q_dev || !gamma_y_dev || !scale_y_dev)
        return PROM_ERR_NULL;
    if (!aligned16(x_dev) || !aligned16(w_packed_dev) || !aligned16(q_dev)) return PROM_ERR_ALIGN;
    if (reinterpret_cast<const void *>(x_dev) == reinterpret_cast<const void *>(q_dev)) return PROM_ERR_ALIGN;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    TcPlan pl;
    const RowMap plain{1, 1, 1, 1, 1};
    if (!tc_shape_plan(m, cin, cout, plain, d, pl, kPlanDynamic)) return PROM_ERR_UNSUPPORTED;
    if (tc_set_attr(d) != PROM_OK) return PROM_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    Conv c;
    c.x = x_dev; c.m = m; c.cin = cin; c.cout = cout; c.map = plain; c.in_rows = m;
    c.w = w_packed_dev; c.y = q_dev; c.st = st;
    // Links of a chain whose first kernel waits before it releases the passes: input, weights and factors
    // are complete when a pass starts, only the maxima are not, so operands are built and the first tiles
    // loaded and multiplied beside the kernel in front.
    c.pdl = tc::kPdlChain;
    c.rq.bias = nullptr; c.rq.shift = nullptr;
    c.rq.mult = reinterpret_cast<const int32_t *>(alpha_dev);     // bit patterns of alpha
    c.rq.act_min = -128; c.rq.act_max = 127;                      // keeps the weights at +-1
    tc_bind(c, pl, nullptr);
    pl.p.dyn = 1;
    pl.p.rows_per_sample = (int)rows_per_sample;
    pl.p.batch = batch;
    pl.p.gamma_x = gamma_x_dev;
    pl.p.gamma_y = gamma_y_dev;
    pl.p.scale_y = scale_y_dev;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, (batch + 127) / 128, 128, 0, st, true);
    const cudaError_t ce = cudaLaunchKernelEx(&cfg, dyn_clear_kernel, gamma_y_dev, batch);
    ++g_launches;
    if (ce != cudaSuccess) return PROM_ERR_CUDA;
    prom_status e = tc_launch_planned(c, pl, 1);
    if (e != PROM_OK) return e;
    return tc_launch_planned(c, pl, 2);
}

prom_status prom_quantize_act_absmax(const float *x_dev, int batch, int64_t per_sample,
                                     int8_t *q_dev, float *gamma_dev, float *scale_dev,
                                     void *cuda_stream)
{
    if (batch < 0 || per_sample < 1 || per_sample > (1ll << 40)) return PROM_ERR_SHAPE;
    if (batch == 0) return PROM_OK;
    if (!x_dev || !q_dev || !gamma_dev || !scale_dev) return PROM_ERR_NULL;
    if (!aligned16(x_dev) || !aligned16(q_dev)) return PROM_ERR_ALIGN;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const float eps = 1e-5f;

    // Fused route: a cluster of CTAs per sample, its slices in shared memory.  The cluster size follows a time
    // model fitted to a B200: every round of resident clusters costs an exchange that grows with the
    // cluster, and the load of an SM's slices at about 100 KB per us.  (190 samples of 125 KB: 7.7 us with
    // clusters of 2, which all fit at once, 10.1 and 11.1 with 1 and 4; 3 samples of 358 KB: 4.3 us with 8,
    // 6.8 with 2.)
    const size_t room = (size_t)d.smem_optin - 4096;
    int cluster = 0, slice = 0;
    long long rounds = 0;
    const long long total_bytes = (long long)batch * per_sample * 4;
    if (per_sample % 16 == 0) {
        double best = 0;
        for (int c = 1, log2c = 0; c <= actq::kMaxCluster; c *= 2, ++log2c) {
            const long long s = ((per_sample + c - 1) / c + 15) / 16 * 16;
            if ((size_t)s * 4 > room) continue;
            long long per_sm = (d.smem_total - 1024) / (s * 4 + 2048);
            if (per_sm > 2048 / actq::kThreads) per_sm = 2048 / actq::kThreads;
            if (per_sm < 1) per_sm = 1;
            const long long at_once = per_sm * d.sms / c > 0 ? per_sm * d.sms / c : 1;
            const long long r = (batch + at_once - 1) / at_once;
            const long long used = ((long long)batch * c + d.sms - 1) / d.sms;
            const double t = (double)r * (2.2 + 0.2 * log2c + (double)(s * 4 * (used < per_sm ? used : per_sm)) / 100e3);
            if (!cluster || t < best) { best = t; cluster = c; slice = (int)s; rounds = r; }
        }
    }
    // Several rounds of clusters run in step, each with its loads exposed; what fits one group of the grouped
    // route below is faster there (192 x 188 KB: 11.3 us against 14.9; 128 x 301 KB: 11.5 against 13.5)
    constexpr long long kOneGroup = 64ll << 20, kGroup = kOneGroup;
    if (rounds > 1 && total_bytes > (24ll << 20) && total_bytes <= kOneGroup) cluster = 0;
    if (cluster) {
        // (whether an SM holds one such CTA or several does not depend on the registers of either form)
        auto *kernel = (size_t)slice * 4 > (size_t)d.smem_total / 2 && rounds > 1 ? actq::act_quant_cluster_kernel<3>
                                                                                    : actq::act_quant_cluster_kernel<0>;
        const cudaError_t attr_err = raise_smem_limit(kernel, d.smem_optin - 4096);
        if (attr_err != cudaSuccess) return cuda_status(attr_err);
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)cluster);       // one cluster, for the occupancy query
        cfg.blockDim = dim3(actq::kThreads);
        cfg.dynamicSmemBytes = (size_t)slice * 4;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        // as many clusters as are resident at once, each walking over its share of the samples
        // (asked once per shape: the query costs tens of microseconds on the host)
        static std::mutex mu;
        static std::map<std::array<long long, 3>, int> known;
        int dev = 0;
        cudaGetDevice(&dev);
        int resident = 0;
        {
            std::lock_guard<std::mutex> lk(mu);
            const std::array<long long, 3> key = {dev, cluster, slice};
            auto it = known.find(key);
            if (it == known.end()) {
                if (cudaOccupancyMaxActiveClusters(&resident, kernel, &cfg) !=
                    cudaSuccess)
                    resident = 0;
                cudaGetLastError();
                known[key] = resident;
            } else {
                resident = it->second;
            }
        }
        if (resident > 0) {
            const int nclusters = resident < batch ? resident : batch;
            cfg.gridDim = dim3((unsigned)(nclusters * cluster));
            attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[1].val.programmaticStreamSerializationAllowed = 1;
            cfg.numAttrs = 2;
            cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, x_dev, batch,
                                               (long long)per_sample, slice, eps, q_dev, gamma_dev,
                                               scale_dev);
            ++g_launches;
            return cuda_status(e);
        }
    }

    // groups of samples, the codes of one behind the maxima of the next
    if (per_sample % 4 == 0) {
        actq::GroupArgs a;
        memset(&a, 0, sizeof(a));
        a.x = x_dev; a.per = per_sample; a.pieces = (per_sample + actq::kPiece - 1) / actq::kPiece;
        a.eps = eps; a.q = q_dev; a.gamma = gamma_dev; a.scale = scale_dev;
        // (groups of up to 64 MB: with 40, or 24, more launches; 6 samples of 23.0 MB 54 us, with 64 47)
        long long per_group = kGroup / (per_sample * 4);
        if (per_group < 1) per_group = 1;
        const long long groups = (batch + per_group - 1) / per_group;
        per_group = (batch + groups - 1) / groups;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        fill_launch_cfg(cfg, attr, (batch + 127) / 128, 128, 0, st, true);
        cudaError_t e = cudaLaunchKernelEx(&cfg, dyn_clear_kernel, gamma_dev, batch);
        ++g_launches;
        for (long long k = 0; k * per_group < batch + per_group && e == cudaSuccess; ++k) {
            auto count = [&](long long first) { return (int)(first < 0 || first >= batch ? 0 : (batch - first < per_group ? batch - first : per_group)); };
            a.first = k == 0;
            a.max_first = (int)(k * per_group < batch ? k * per_group : 0); a.max_count = count(k * per_group);
            a.q_first = k ? (int)((k - 1) * per_group) : 0; a.q_count = k ? count((k - 1) * per_group) : 0;
            // blocks for about two pieces per warp and pass, at most two per SM
            const long long most = a.pieces * (a.max_count > a.q_count ? a.max_count : a.q_count);
            long long blocks = (most + 31) / 32;
            if (blocks > 2 * d.sms) blocks = 2 * d.sms;
            fill_launch_cfg(cfg, attr, (int)blocks, actq::kGroupThreads, 0, st, true);
            e = cudaLaunchKernelEx(&cfg, groups > 1 ? actq::act_group_kernel<true> : actq::act_group_kernel<false>, a);
            ++g_launches;
        }
        return cuda_status(e);
    }

    // two passes
    if (cudaMemsetAsync(gamma_dev, 0, sizeof(float) * (size_t)batch, st) != cudaSuccess) return PROM_ERR_CUDA;
    long long bx = (per_sample + actq::kThreads * 8 - 1) / (actq::kThreads * 8);
    const long long cap = (long long)d.sms * 8 / batch + 1;
    if (bx > cap) bx = cap;
    if (bx < 1) bx = 1;
    const dim3 grid((unsigned)bx, (unsigned)batch);
    if (batch > 65535) return PROM_ERR_SHAPE;
    actq::act_absmax_kernel<<<grid, actq::kThreads, 0, st>>>(x_dev, (long long)per_sample, gamma_dev);
    ++g_launches;
    actq::act_quant_kernel<<<grid, actq::kThreads, 0, st>>>(x_dev, (long long)per_sample, eps, gamma_dev, q_dev,
                                                            scale_dev);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

prom_status prom_requant_from_scale(double scale, int32_t *mult, int8_t *shift)
{
    if (!mult || !shift) return PROM_ERR_NULL;
    if (!(scale > 0.0) || scale >= 1.0) return PROM_ERR_BAD_REQUANT;
    // scale = f * 2^(e+1) with f in [0.5, 1): mult = round(f * 2^31), shift = -(e+1)
    int e = ilogb(scale);                        // floor(log2(scale)), <= -1
    int sh = -(e + 1);
    double m = nearbyint(scalbn(scale, 31 + sh));
    if (m >= 2147483648.0) { m = 1073741824.0; --sh; }
    if (sh < 0 || sh > 31) return PROM_ERR_BAD_REQUANT;
    *mult = (int32_t)m;
    *shift = (int8_t)sh;
    return PROM_OK;
}

prom_status prom_pw_conv_i8(const int8_t *x_dev, int64_t m, int cin, const uint8_t *w_packed_dev,
                            int cout, const prom_requant *rq, int8_t *y_dev, prom_variant variant,
                            void *cuda_stream)
{
    // an empty matrix has no rows to read or write: its pointers may be anything
    if (m == 0 && cin >= 1 && cin <= 4096 && cout >= 1 && cout <= 4096 && w_packed_dev && rq)
        return check_requant(rq);
    prom_status s = check_conv(x_dev, m, cin, w_packed_dev, cout, rq, y_dev);
    if (s != PROM_OK) return s;
    Conv c;
    c.x = x_dev; c.m = m; c.cin = cin; c.cout = cout;
    c.map = RowMap{1, 1, 1, 1, 1};
    c.in_rows = m;
    c.w = w_packed_dev; c.rq = *rq; c.y = y_dev;
    c.st = static_cast<cudaStream_t>(cuda_stream);
    return run_conv(c, variant);
}

// ---- one layer with operands prepared ahead of the call --------------------------------------
static Conv prepared_conv(long long m, int cin, int cout)
{
    Conv c;
    c.m = m; c.cin = cin; c.cout = cout; c.map = RowMap{1, 1, 1, 1, 1}; c.in_rows = m;
    return c;
}
static bool prepared_plan(long long m, int cin, int cout, const DeviceInfo &d, TcPlan &pl)
{
    return m > 0 && tc_shape_plan(m, cin, cout, RowMap{1, 1, 1, 1, 1}, d, pl, kPlanPrepared);
}
// Whether the prepared form of a layer is the row-resident kernel's.
static bool prepared_wide(const Conv &c, const DeviceInfo &d, WidePlan &pl)
{
    const int mode = g_wide_mode.load();
    bool worth = false;
    if (mode == 1 || !wide_plan(c, d, pl, worth)) return false;
    return mode == 2 || wide_prepared_worth(c, d);
}

size_t prom_pw_prepared_bytes(int64_t m, int cin, int cout)
{
    if (m < 1 || cin < 1 || cin > 4096 || cout < 1 || cout > 4096) return 0;
    DeviceInfo d = device_info();
    if (!d.ok) { d.sms = 148; d.smem_optin = 232448; d.smem_total = 233472; d.ok = true; }
    WidePlan wp;
    if (prepared_wide(prepared_conv(m, cin, cout), d, wp)) return wide_operand_bytes(wp);
    TcPlan pl;
    if (!prepared_plan(m, cin, cout, d, pl)) return 0;
    return round256((size_t)pl.p.groups * pl.p.image_stride);
}

prom_status prom_pw_prepare(int64_t m, int cin, const uint8_t *w_packed_dev, int cout, const prom_requant *rq,
                            void *prepared_dev, size_t prepared_bytes, void *cuda_stream)
{
    if (!w_packed_dev || !prepared_dev) return PROM_ERR_NULL;
    prom_status e = check_requant(rq);
    if (e != PROM_OK) return e;
    if (m < 1 || cin < 1 || cin > 4096 || cout < 1 || cout > 4096) return PROM_ERR_SHAPE;
    if (!aligned16(w_packed_dev) || !aligned16(prepared_dev)) return PROM_ERR_ALIGN;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    Conv c = prepared_conv(m, cin, cout);
    c.w = w_packed_dev; c.rq = *rq; c.st = static_cast<cudaStream_t>(cuda_stream);
    WidePlan wp;
    if (prepared_wide(c, d, wp)) {
        if (prepared_bytes < wide_operand_bytes(wp)) return PROM_ERR_WORKSPACE;
        return launch_wide_prep(c, wp, static_cast<uint8_t *>(prepared_dev));
    }
    TcPlan pl;
    if (!prepared_plan(m, cin, cout, d, pl)) return PROM_ERR_UNSUPPORTED;
    if (prepared_bytes < round256((size_t)pl.p.groups * pl.p.image_stride)) return PROM_ERR_WORKSPACE;
    if (tc_set_attr(d) != PROM_OK) return PROM_ERR_CUDA;
    tc_bind(c, pl, static_cast<uint8_t *>(prepared_dev));
    tc::PrepTable t;
    memset(&t, 0, sizeof(t));
    int ctas = 0;
    size_t smem = 0;
    prep_add(t, pl.p, ctas, smem);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch_cfg(cfg, attr, ctas, tc::kPrepThreads, smem, c.st, true);
    const cudaError_t le = cudaLaunchKernelEx(&cfg, tc::tc_prep_kernel, t);
    ++g_launches;
    return cuda_status(le);
}

prom_status prom_pw_conv_i8_prepared(const int8_t *x_dev, int64_t m, int cin, int cout, const void *prepared_dev,
                                     int act_min, int act_max, int8_t *y_dev, void *cuda_stream)
{
    if (act_min < -128 || act_max > 127 || act_min > act_max) return PROM_ERR_BAD_REQUANT;
    if (cin < 1 || cin > 4096 || cout < 1 || cout > 4096 || m < 0 || m > (1ll << 40)) return PROM_ERR_SHAPE;
    if (m == 0) return PROM_OK;
    if (!x_dev || !prepared_dev || !y_dev) return PROM_ERR_NULL;
    if (!aligned16(x_dev) || !aligned16(prepared_dev) || !aligned16(y_dev)) return PROM_ERR_ALIGN;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    Conv c = prepared_conv(m, cin, cout);
    c.x = x_dev; c.y = y_dev; c.st = static_cast<cudaStream_t>(cuda_stream);
    c.rq = prom_requant{nullptr, nullptr, nullptr, act_min, act_max};
    WidePlan wp;
    if (prepared_wide(c, d, wp)) return launch_wide_conv(c, wp, const_cast<uint8_t *>(static_cast<const uint8_t *>(prepared_dev)));
    TcPlan pl;
    if (!prepared_plan(m, cin, cout, d, pl)) return PROM_ERR_UNSUPPORTED;
    if (tc_set_attr(d) != PROM_OK) return PROM_ERR_CUDA;
    tc_bind(c, pl, const_cast<uint8_t *>(static_cast<const uint8_t *>(prepared_dev)));
    return tc_launch_planned(c, pl);
}

prom_status prom_pw_conv_i8_res(const int8_t *x_dev, int64_t m, int cin, const uint8_t *w_packed_dev,
                                int cout, const prom_requant *rq, const int8_t *res_dev,
                                int8_t *y_dev, prom_variant variant, void *cuda_stream)
{
    if (m == 0 && cin >= 1 && cin <= 4096 && cout >= 1 && cout <= 4096 && w_packed_dev && rq)
        return check_requant(rq);
    prom_status s = check_conv(x_dev, m, cin, w_packed_dev, cout, rq, y_dev);
    if (s != PROM_OK) return s;
    if (!res_dev) return PROM_ERR_NULL;
    if (!aligned16(res_dev)) return PROM_ERR_ALIGN;
    Conv c;
    c.x = x_dev; c.m = m; c.cin = cin; c.cout = cout;
    c.map = RowMap{1, 1, 1, 1, 1};
    c.in_rows = m;
    c.w = w_packed_dev; c.rq = *rq; c.y = y_dev;
    c.st = static_cast<cudaStream_t>(cuda_stream);
    c.res = res_dev;
    return run_conv(c, variant);
}

prom_status prom_pw_conv_i8_acc32(const int8_t *x_dev, int64_t m, int cin,
                                  const uint8_t *w_packed_dev, int cout, int32_t *acc_dev,
                                  void *cuda_stream)
{
    if (!x_dev || !w_packed_dev || !acc_dev) return PROM_ERR_NULL;
    if (m < 0 || cin < 1 || cin > 4096 || cout < 1 || cout > 4096) return PROM_ERR_SHAPE;
    if (m == 0) return PROM_OK;
    Conv c;
    c.x = x_dev; c.m = m; c.cin = cin; c.cout = cout;
    c.map = RowMap{1, 1, 1, 1, 1};
    c.in_rows = m;
    c.w = w_packed_dev;
    c.rq = prom_requant{nullptr, nullptr, nullptr, 0, 127};
    c.y = nullptr;
    c.st = static_cast<cudaStream_t>(cuda_stream);
    return launch_naive(c, acc_dev);
}

prom_status prom_pw_conv_i8_host(const int8_t *x_host, int64_t m, int cin,
                                 const uint8_t *w_packed_dev, int cout, const prom_requant *rq,
                                 int8_t *y_host, void *workspace_dev, size_t workspace_bytes,
                                 prom_variant variant, void *cuda_stream)
{
    if (!x_host || !y_host || !workspace_dev) return PROM_ERR_NULL;
    if (m < 0 || cin < 1 || cout < 1) return PROM_ERR_SHAPE;
    size_t xb = round256((size_t)m * cin), yb = round256((size_t)m * cout);
    if (workspace_bytes < xb + yb) return PROM_ERR_WORKSPACE;
    if (!aligned16(workspace_dev)) return PROM_ERR_ALIGN;
    int8_t *xd = static_cast<int8_t *>(workspace_dev);
    int8_t *yd = xd + xb;
    prom_status s = check_conv(xd, m, cin, w_packed_dev, cout, rq, yd);
    if (s != PROM_OK) return s;
    if (m == 0) return PROM_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemcpyAsync(xd, x_host, (size_t)m * cin, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return PROM_ERR_CUDA;
    s = prom_pw_conv_i8(xd, m, cin, w_packed_dev, cout, rq, yd, variant, cuda_stream);
    if (s != PROM_OK) return s;
    return cuda_status(cudaMemcpyAsync(y_host, yd, (size_t)m * cout, cudaMemcpyDeviceToHost, st));
}

size_t prom_layer_seq_workspace_bytes(const prom_layer *layers, int n, int batch, int h0, int w0)
{
    SeqShape s;
    if (!seq_shapes(layers, n, batch, h0, w0, s)) return 0;
    DeviceInfo d = device_info();
    SeqLayout lay;
    seq_layout(layers, n, s, d, true, lay);
    if (!lay.chains.empty()) return lay.with_chains();
    const size_t blocks = lay.blocks.empty() ? 0 : lay.with_blocks();
    if (blocks) {                 // room for one launch per layer too: what the call falls back on
        lay = SeqLayout();
        seq_layout(layers, n, s, d, true, lay, true, false);
    }
    const size_t plain = lay.img_total ? lay.with_images() : lay.base();
    return blocks > plain ? blocks : plain;
}

prom_status prom_pw_layer_seq(const prom_layer *layers, int n, const int8_t *x0_dev, int batch,
                              int h0, int w0, void *workspace_dev, size_t workspace_bytes,
                              int8_t *y_out_dev, prom_variant variant, void *cuda_stream)
{
    if (!layers || !x0_dev || !y_out_dev) return PROM_ERR_NULL;
    if (!aligned16(x0_dev) || !aligned16(y_out_dev)) return PROM_ERR_ALIGN;
    return run_seq(layers, n, x0_dev, batch, h0, w0, workspace_dev, workspace_bytes, y_out_dev,
                   variant, static_cast<cudaStream_t>(cuda_stream));
}

size_t prom_layer_seq_host_workspace_bytes(const prom_layer *layers, int n, int batch, int h0,
                                           int w0)
{
    SeqShape s;
    if (!seq_shapes(layers, n, batch, h0, w0, s)) return 0;
    const size_t core = round256(prom_layer_seq_workspace_bytes(layers, n, batch, h0, w0));
    size_t xin = round256((size_t)batch * h0 * w0 * layers[0].cin);
    size_t yout = round256((size_t)s.m[n - 1] * layers[n - 1].cout);
    return core + xin + yout;
}

prom_status prom_pw_layer_seq_host(const prom_layer *layers, int n, const int8_t *x0_host,
                                   int batch, int h0, int w0, void *workspace_dev,
                                   size_t workspace_bytes, int8_t *y_out_host, prom_variant variant,
                                   void *cuda_stream)
{
    if (!layers || !x0_host || !y_out_host || !workspace_dev) return PROM_ERR_NULL;
    if (!aligned16(workspace_dev)) return PROM_ERR_ALIGN;
    SeqShape s;
    if (!seq_shapes(layers, n, batch, h0, w0, s)) return PROM_ERR_SHAPE;
    const size_t core = round256(prom_layer_seq_workspace_bytes(layers, n, batch, h0, w0));
    size_t xin_raw = (size_t)batch * h0 * w0 * layers[0].cin;
    size_t yout_raw = (size_t)s.m[n - 1] * layers[n - 1].cout;
    size_t xin = round256(xin_raw), yout = round256(yout_raw);
    if (workspace_bytes < core + xin + yout) return PROM_ERR_WORKSPACE;
    int8_t *base = static_cast<int8_t *>(workspace_dev);
    int8_t *xd = base + core, *yd = xd + xin;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemcpyAsync(xd, x0_host, xin_raw, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return PROM_ERR_CUDA;
    prom_status e = run_seq(layers, n, xd, batch, h0, w0, base, core, yd, variant, st);
    if (e != PROM_OK) return e;
    return cuda_status(cudaMemcpyAsync(y_out_host, yd, yout_raw, cudaMemcpyDeviceToHost, st));
}

prom_status prom_pw_conv_i8_addsub_static(const int8_t *x_dev, int64_t m, int cin,
                                          const uint8_t *w_packed_dev, int cout,
                                          const prom_requant *rq, int8_t *y_dev,
                                          void *cuda_stream)
{
    // an empty matrix has no rows to read or write: its pointers may be anything
    if (m == 0 && cin >= 1 && cin <= 4096 && cout >= 1 && cout <= 4096 && w_packed_dev && rq)
        return check_requant(rq);
    prom_status s = check_conv(x_dev, m, cin, w_packed_dev, cout, rq, y_dev);
    if (s != PROM_OK) return s;
    if (cin > addsub::kMaxCin) return PROM_ERR_UNSUPPORTED;
    if (addsub::scratch_bytes(cout, cin) > (size_t)PROM_STATIC_SCRATCH_BYTES)
        return PROM_ERR_WORKSPACE;
    if (m == 0) return PROM_OK;
    uint8_t *scratch = static_scratch_address();
    if (!scratch) return PROM_ERR_CUDA;
    return addsub::launch_on(x_dev, m, cin, RowMap{1, 1, 1, 1, 1}, w_packed_dev, cout, *rq, y_dev,
                             scratch, static_cast<cudaStream_t>(cuda_stream), g_launches);
}

prom_status prom_last_device_status(void *cuda_stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    unsigned int v = 0;
    if (cudaMemcpyFromSymbolAsync(&v, g_status, sizeof(v), 0, cudaMemcpyDeviceToHost, st) !=
        cudaSuccess)
        return PROM_ERR_CUDA;
    unsigned int zero = 0;
    if (cudaMemcpyToSymbolAsync(g_status, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice, st) !=
        cudaSuccess)
        return PROM_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return PROM_ERR_CUDA;
    return static_cast<prom_status>(v);
}

uint64_t prom_launch_count(void) { return g_launches.load(); }

void prom_debug_tc_plan_shape(int64_t m, int cin, int cout, int stride, int fold, int nt, int groups,
                              int occ, int stages)
{
    std::lock_guard<std::mutex> lk(g_shape_tune_mu);
    const std::array<long long, 4> key = {m, cin, cout, stride};
    if (!fold && !nt && !groups && !occ && !stages) g_shape_tune.erase(key);
    else g_shape_tune[key] = TcTune{fold, nt, groups, occ, stages};
    g_tuned.store(true);
}

void prom_debug_tc_plan(int fold, int nt, int groups, int occ, int stages)
{
    std::lock_guard<std::mutex> lk(g_shape_tune_mu);
    g_tune = TcTune{fold, nt, groups, occ, stages};
    g_tuned.store(fold || nt || groups || occ || stages || !g_shape_tune.empty());
}

prom_status prom_debug_wait_timeout(uint64_t limit_ns, int *gave_up_dev, void *cuda_stream)
{
    if (limit_ns < 1000 || limit_ns > 100000000ull) return PROM_ERR_SHAPE;
    tc::wait_timeout_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        (unsigned long long)limit_ns, gave_up_dev);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

prom_status prom_debug_i8_mma_rate(int iters, long long *cycles_dev, int cycles_len, int *grid_out,
                                   void *cuda_stream)
{
    if (!cycles_dev || !grid_out) return PROM_ERR_NULL;
    if (iters < 1 || iters > (1 << 20)) return PROM_ERR_SHAPE;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    if (cycles_len < d.sms) return PROM_ERR_WORKSPACE;
    if (raise_smem_limit(peak::i8_mma_rate_kernel, peak::kMmaSmem) != cudaSuccess) return PROM_ERR_CUDA;
    *grid_out = d.sms;
    peak::i8_mma_rate_kernel<<<d.sms, peak::kMmaThreads, peak::kMmaSmem,
                               static_cast<cudaStream_t>(cuda_stream)>>>(iters, cycles_dev);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

prom_status prom_debug_alu_rate(int op, int iters, int *sink_dev, long long *cycles_dev,
                                int cycles_len, int *grid_out, void *cuda_stream)
{
    if (!sink_dev || !cycles_dev || !grid_out) return PROM_ERR_NULL;
    if (op < 0 || op > 6 || iters < 1 || iters > (1 << 24)) return PROM_ERR_SHAPE;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    const int grid = 2 * d.sms;
    if (cycles_len < grid) return PROM_ERR_WORKSPACE;
    *grid_out = grid;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (op == 0) peak::alu_rate_kernel<0><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    else if (op == 1) peak::alu_rate_kernel<1><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    else if (op == 2) peak::alu_rate_kernel<2><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    else if (op == 3) peak::alu_rate_kernel<3><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    else if (op == 4) peak::alu_rate_kernel<4><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    else if (op == 5) peak::alu_rate_kernel<5><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    else peak::alu_rate_kernel<6><<<grid, peak::kAluThreads, 0, st>>>(iters, 1, sink_dev, cycles_dev);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

prom_status prom_debug_mma_issue_rate(int n, int warps, int iters, long long *cycles_dev, int cycles_len,
                                      int *grid_out, void *cuda_stream)
{
    if (!cycles_dev || !grid_out) return PROM_ERR_NULL;
    if (n < 16 || n > 256 || (n & 15) || warps < 1 || warps > 4 || iters < 1 || iters > (1 << 20))
        return PROM_ERR_SHAPE;
    if (warps * 2 * (n > 64 ? n : 64) > 512) return PROM_ERR_SHAPE;     // tensor-memory columns
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    if (cycles_len < 4 * d.sms) return PROM_ERR_WORKSPACE;
    *grid_out = d.sms;
    if (raise_smem_limit(peak::mma_issue_rate_kernel, peak::kMmaSmem) != cudaSuccess) return PROM_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemsetAsync(cycles_dev, 0, sizeof(long long) * 4 * (size_t)d.sms, st) != cudaSuccess) return PROM_ERR_CUDA;
    peak::mma_issue_rate_kernel<<<d.sms, peak::kMmaThreads, peak::kMmaSmem, st>>>(iters, n, warps, cycles_dev);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

prom_status prom_debug_l2_copy_rate(const void *region_dev, uint64_t region_bytes, int iters, int stages,
                                    long long *cycles_dev, int cycles_len, int *grid_out, void *cuda_stream)
{
    if (!region_dev || !cycles_dev || !grid_out) return PROM_ERR_NULL;
    if (!aligned16(region_dev)) return PROM_ERR_ALIGN;
    if (region_bytes < peak::kCopyBytes || region_bytes % peak::kCopyBytes || iters < 1 || iters > (1 << 20) ||
        stages < 1 || stages > peak::kCopyMaxStages)
        return PROM_ERR_SHAPE;
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    if (cycles_len < d.sms) return PROM_ERR_WORKSPACE;
    *grid_out = d.sms;
    const int smem = peak::kCopyMaxStages * (int)peak::kCopyBytes + 256;
    if (raise_smem_limit(peak::l2_copy_rate_kernel, smem) != cudaSuccess) return PROM_ERR_CUDA;
    peak::l2_copy_rate_kernel<<<d.sms, 32, smem, static_cast<cudaStream_t>(cuda_stream)>>>(
        static_cast<const uint8_t *>(region_dev), (unsigned long long)region_bytes, iters, stages, cycles_dev);
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

prom_status prom_debug_mma_beside(int mode, int iters, int nwarps, int stages, const void *region_dev,
                                  uint64_t region_bytes, long long *out_dev, int out_len, int *grid_out,
                                  void *cuda_stream)
{
    if (!out_dev || !grid_out) return PROM_ERR_NULL;
    if ((mode != 0 && mode != 1) || iters < 1 || iters > (1 << 20)) return PROM_ERR_SHAPE;
    if (mode == 0) {
        if (stages < 0 || stages > 3) return PROM_ERR_SHAPE;
        if (stages > 0) {
            if (!region_dev) return PROM_ERR_NULL;
            if (!aligned16(region_dev)) return PROM_ERR_ALIGN;
            if (region_bytes < peak::kCopyBytes || region_bytes % peak::kCopyBytes) return PROM_ERR_SHAPE;
        }
    } else if ((nwarps != 4 && nwarps != 8 && nwarps != 16) || (stages != 0 && stages != 1)) {
        return PROM_ERR_SHAPE;
    }
    DeviceInfo d = device_info();
    if (!d.ok) return PROM_ERR_CUDA;
    if (out_len < 8 * d.sms) return PROM_ERR_WORKSPACE;
    *grid_out = d.sms;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemsetAsync(out_dev, 0, sizeof(long long) * 8 * (size_t)d.sms, st) != cudaSuccess) return PROM_ERR_CUDA;
    const uint8_t *src = static_cast<const uint8_t *>(region_dev);
    if (mode == 0) {
        if (raise_smem_limit(peak::beside_mma_kernel<0>, peak::kBesideSmem) != cudaSuccess) return PROM_ERR_CUDA;
        peak::beside_mma_kernel<0><<<d.sms, peak::kBesideThreads, peak::kBesideSmem, st>>>(
            iters, 0, stages, src, (unsigned long long)region_bytes, out_dev);
    } else {
        if (raise_smem_limit(peak::beside_mma_kernel<1>, peak::kBesideSmem) != cudaSuccess) return PROM_ERR_CUDA;
        peak::beside_mma_kernel<1><<<d.sms, peak::kBesideThreads, peak::kBesideSmem, st>>>(
            iters, nwarps, stages, src, (unsigned long long)region_bytes, out_dev);
    }
    ++g_launches;
    return cuda_status(cudaGetLastError());
}

void prom_debug_seq_order(int alternate) { g_seq_snake.store(alternate ? 1 : 0); }
void prom_debug_seq_chain(int mode) { g_seq_chain.store(mode == 2 ? 2 : (mode ? 1 : 0)); }

void prom_debug_seq_block(int mode, int rows, int split)
{
    g_block_mode.store(mode < 0 || mode > 2 ? 0 : mode);
    g_block_rows.store(rows);
    g_block_split.store(split);
}
void prom_debug_dw_variant(int variant) { g_dw_variant.store(variant < 0 || variant > 2 ? 0 : variant); }

void prom_debug_tc_wide(int mode, int blocks)
{
    g_wide_mode.store(mode < 0 || mode > 2 ? 0 : mode);
    g_wide_nb.store(blocks == 1 || blocks == 2 ? blocks : 0);
}

int64_t prom_debug_layer_seq_output_offset(const prom_layer *layers, int n, int batch, int h0, int w0,
                                           int layer, int *chained)
{
    SeqShape s;
    if (!seq_shapes(layers, n, batch, h0, w0, s) || layer < 0 || layer >= n - 1) return -1;
    DeviceInfo d = device_info();
    SeqLayout lay;
    seq_layout(layers, n, s, d, true, lay);
    const bool in_chain = lay.chain_of[layer] >= 0;
    if (chained) *chained = in_chain ? 1 : 0;
    if (in_chain) {
        const ChainPlan &c = lay.chains[lay.chain_of[layer]];
        if (c.kind == 1 && layer != c.last) return -2;      // never written: it stays in shared memory
        return (int64_t)(round256(lay.with_images()) + lay.cbuf_off[layer]);
    }
    if (lay.block_of[layer] >= 0 && lay.block_of[layer + 1] == lay.block_of[layer]) {
        if (chained) *chained = 1;
        return -2;                                          // a block's expanded tensor is never written
    }
    return lay.region[layer] ? (int64_t)lay.ra : 0;
}

int prom_debug_once_per_device(int device, int key)
{
    static OncePerDevice table;
    return table.first(device, reinterpret_cast<const void *>((intptr_t)key)) ? 1 : 0;
}

int prom_debug_tc_plan_query(int64_t m, int cin, int cout, int *out9)
{
    if (!out9) return 0;
    DeviceInfo d = device_info();
    if (!d.ok) {
        // no device to ask: the plan for a B200 as shipped (148 SMs, 227 KB of shared memory a
        // CTA can opt into, 228 KB per SM), so that the planner can be exercised anywhere
        d.sms = 148; d.smem_optin = 232448; d.smem_total = 233472; d.ok = true;
    }
    TcPlan pl;
    if (!tc_shape_plan(m, cin, cout, RowMap{1, 1, 1, 1, 1}, d, pl)) return 0;
    const tc::Params &p = pl.p;
    out9[0] = p.fold; out9[1] = p.nt; out9[2] = p.groups; out9[3] = pl.grid; out9[4] = p.stages;
    out9[5] = p.nbuf; out9[6] = (int)pl.smem; out9[7] = p.cw; out9[8] = (int)(pl.est_us * 100);
    return 1;
}

void prom_shutdown(void)
{
    addsub::release_cache();
    wide_release_cache();
}

const char *prom_status_string(prom_status s)
{
    switch (s) {
    case PROM_OK: return "ok";
    case PROM_ERR_NULL: return "null pointer";
    case PROM_ERR_SHAPE: return "bad shape";
    case PROM_ERR_ALIGN: return "misaligned pointer";
    case PROM_ERR_BAD_WEIGHT: return "weight outside {-1,0,+1}";
    case PROM_ERR_BAD_REQUANT: return "requantisation constants out of range";
    case PROM_ERR_WORKSPACE: return "workspace too small";
    case PROM_ERR_UNSUPPORTED: return "variant does not support this shape";
    case PROM_ERR_CUDA: return "CUDA call failed";
    case PROM_ERR_TIMEOUT: return "device-side wait ran out";
    default: return "unknown status";
    }
}

}  // extern "C"
