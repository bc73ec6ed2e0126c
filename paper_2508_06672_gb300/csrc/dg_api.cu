// dg_api.cu -- host implementation of the C ABI declared in include/dg.h.
//
// The context owns every device buffer of the hot path: shard ECEF [3][G],
// ephemerides [K][12], per-snapshot captures (raw format, not widened), the
// per-snapshot surfaces [K][G] (scratch for the ordered accumulation), the
// argmax scratch and the refinement buffers. All allocation is
// stream-ordered (cudaMallocAsync / cudaFreeAsync) on the context's stream.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstring>
#include <list>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "dg_internal.cuh"

using namespace dg;

namespace {

thread_local std::string g_thread_error;

struct Step {
    int fmt = -1;
    int64_t n = 0;
    void *y1 = nullptr, *y2 = nullptr;
    size_t cap = 0;  // bytes per receiver buffer
    bool loaded = false;
};

struct TimedLaunch {
    int cls;
    cudaEvent_t a, b;
};

struct CdftLayout {  // batches and bucket / group bases of one grid size
    struct Batch {
        int k0, S, base;      // snapshots k0 .. k0 + S - 1; offset of its bases
        int64_t nbt, groups;  // lag slots and combine groups (upper bounds)
    };
    int64_t G = -1;
    int nseg = 0;           // segments of samples (direct surfaces)
    bool direct = false;    // lag groups of direct surfaces
    std::vector<int> fmts;  // the captures' formats (a batch of the contraction has one)
    double diam = 0.0;      // grid diameter bound the lag slots were sized for
    std::vector<Batch> batches;
    int s_max = 0;
    int64_t nbt_max = 0, groups_max = 0;
    int *bbase = nullptr, *gbase = nullptr;  // device, per batch: [S + 1] each
};

struct CdftRun {  // one chunked-DFT surface, phase by phase (run_surface_cdft)
    GridDev gd{};
    const double *xyz = nullptr;
    int64_t G = 0;
    void *surf = nullptr, *out = nullptr;
    bool refine = false, mma = false;
    CdftLayout *L = nullptr;
    std::vector<int> Ms;  // chunk of each batch of snapshots
};

struct GridRange {  // what a grid's nodes can take in one snapshot
    double d_lo, d_hi;    // D (samples)
    double nu_lo, nu_hi;  // FDOA (cycles per sample)
    double rho, sep, vel; // least range (0: none), receivers' separation and speed
    double row_m, col_m;  // longest step between neighbouring rows and columns
};

struct MapPlan {  // shapes of the delay-Doppler maps of the main grid (dg_map.cu)
    uint64_t gen = 0;   // steps_gen it was made for (0: none)
    bool ok = false;    // the grid and captures suit the maps
    int logn = 0, Mb = 0, Cmax = 0, P = 0, Q = 0, LT = 0, ntile = 0, NLpad = 0, S = 0;
    bool c64 = false;
    int chunk_min = 0, chunk_max = 0;  // what dg_cdft_chunks reports
    int64_t rows = 0;                  // (lag, block) pairs of one surface
    double xnode[kMapMaxNodes] = {};
    PolyShape poly{};
};

struct MapBufs {  // their device tables and scratch, grown on demand
    MapSnap *snap = nullptr;
    float2 *tw = nullptr, *F2 = nullptr, *U = nullptr, *X = nullptr, *phase = nullptr;
    float *T = nullptr, *fit = nullptr, *coef = nullptr;
    int fit_rows = 0;  // tile shape fit is for
    size_t fit_cap = 0, coef_cap = 0;
    int *bad = nullptr;
    size_t snap_cap = 0, tw_cap = 0, F2_cap = 0, U_cap = 0, X_cap = 0, phase_cap = 0, T_cap = 0, bad_cap = 0;
    int tw_logn = 0, T_P = 0, T_Q = 0;  // what tw and T hold
};

struct BatchHold {  // a batch's replays read a context's buffers
    cudaEvent_t last = nullptr;  // recorded behind its latest replay
    uint64_t gen = 0;            // the context's steps_gen that the replays need
    std::atomic<bool> alive{true};
    double fill = 0.0;           // tiles_faster: tiles per SM of the whole batch
};

struct LagRule {  // tiles_faster's answer for one grid
    GridDev g{};
    double fill = 0.0;
    bool known = false, tiles = false;
};

struct CdftBufs {  // chunked-DFT scratch, grown on demand
    int *lr = nullptr;
    CdftLayout main_layout, loc_layout;
    CdftLayout dmain_layout, dloc_layout;  // the direct path's lag groups
    std::list<CdftLayout> kept;            // layouts of other shapes, while a captured step may read their tables
    LagRule dmain_rule, dloc_rule;
    double fill = 0.0;                     // while a batch is being captured: BatchHold::fill
    uint64_t no_sort = 0;                  // steps_gen at which the sort found no memory
    float2 *part = nullptr;                // and its segments' sums
    size_t part_cap = 0;
    std::vector<double> main_span;  // FDOA span estimates per snapshot (main grid)
    std::vector<double> main_lags;  // and lag-count estimates
    std::vector<GridRange> main_range;  // and lag / FDOA bounds
    CdftRun main_run;               // the main surface's last run (its batches' arguments)
    int *layout = nullptr, *Mcs = nullptr;
    unsigned long long *work = nullptr;
    unsigned *nur = nullptr;
    float *nubase = nullptr;
    size_t s_cap = 0;
    int *candL = nullptr, *order = nullptr;
    float *candNu = nullptr, *nuS = nullptr;
    float *candMu = nullptr, *muS = nullptr;  // Lagrange4: fractional delays
    size_t mu_cap = 0;
    int *need = nullptr;
    size_t sg_cap = 0;
    int4 *g2b = nullptr;
    size_t g2b_cap = 0;
    float *xyzf = nullptr;
    size_t xyzf_cap = 0;
    float *ephf = nullptr;
    size_t ephf_cap = 0;
    int *count = nullptr, *offs = nullptr, *subcnt = nullptr;
    size_t nb_cap = 0;
    float *delta = nullptr;
    float2 *V = nullptr;
    size_t v_cap = 0;
    float *W = nullptr;
    size_t w_cap = 0;
    int *tbase = nullptr, *hbase = nullptr;
    void *btab = nullptr;
    size_t btab_cap = 0;
};

struct LocalGrid {  // refinement buffers, grown on demand
    double *xyz = nullptr;
    void *surf = nullptr;
    void *cost = nullptr;
    size_t g_cap = 0;
};

struct CoarseBufs {  // coarse delay-Doppler maps (dg_coarse_maps), grown on demand
    int *lag = nullptr;
    float *nu = nullptr;
    int *lmm = nullptr;
    unsigned long long *nmm = nullptr;
    CoarseStep *st = nullptr;
    float2 *P = nullptr, *tw = nullptr, *F2 = nullptr;
    float *A = nullptr, *pool = nullptr;
    float4 *turn = nullptr;
    MapSnap *snap = nullptr;
    int *bad = nullptr;
    double *part = nullptr;
    size_t lag_cap = 0, nu_cap = 0, lmm_cap = 0, nmm_cap = 0, st_cap = 0, P_cap = 0, A_cap = 0, part_cap = 0;
    size_t tw_cap = 0, F2_cap = 0, pool_cap = 0, turn_cap = 0, snap_cap = 0, bad_cap = 0;
    int tw_logn = 0;  // what tw holds
    int Q = 0, M = 0, nlag_cap = 0, nb_max = 0;  // shape of the last maps (Q = 0: none yet)
};

struct PastGrid {  // host bounds of a grid the context had (grid_bounds_switch)
    dg_grid grid;
    std::vector<double> span, lags;
    std::vector<GridRange> range;
};

}  // namespace

struct dg_ctx {
    std::vector<PastGrid> past;  // at most four
    dg_grid grid{};
    dg_options opt{};
    int K = 0;
    double fs = 0, fc = 0, lambda = 0;
    cudaStream_t stream = nullptr;
    int device = 0;
    int sm_count = 1;
    GridDev gd{};
    int64_t G = 0;
    int64_t xyz_cap = 0;                // nodes the ECEF buffer holds
    ArgmaxResult *reg_res = nullptr;    // dg_search_regions: argmax per region (device)
    ArgmaxResult *reg_host = nullptr;   // pinned mirror
    size_t reg_cap = 0;
    double *xyz = nullptr;
    GridStep *gstep = nullptr;          // angular steps of the grid, of the refinement grid (device)
    double *eph = nullptr;
    std::vector<dg_ephem> eph_host;
    std::vector<Step> steps;
    StepDesc *steps_d = nullptr;
    std::vector<StepDesc> steps_h;
    bool steps_dirty = true;
    void *surf = nullptr;
    size_t surf_bytes = 0;
    void *amax_tmp = nullptr;
    size_t amax_tmp_bytes = 0;
    ArgmaxResult *amax_res = nullptr;
    ArgmaxResult *amax_host = nullptr;  // pinned
    int64_t *det_cand = nullptr;
    DetectPeak *det_out = nullptr, *det_host = nullptr;
    int reg_n = 0;  // regions of the last search, their records in reg_host
    unsigned *err_d = nullptr;
    unsigned *err_h = nullptr;          // pinned mirror
    LocalGrid loc;
    CdftBufs cd;
    MapPlan mp;
    MapBufs mb, mr;         // main surface; refinement
    double *reg_xyz = nullptr;          // dg_search_regions: ECEF of the regions searched together
    GridDev *reg_grids = nullptr;
    GridStep *reg_steps = nullptr;
    size_t reg_xyz_cap = 0, reg_grids_cap = 0, reg_steps_cap = 0;
    bool last_map = false;  // the last CDFT surface came from the maps
    CoarseBufs co;
    int cd_chunk_min = 0, cd_chunk_max = 0;              // chunks it used
    // whole-step CUDA graph (dg_graph_*)
    ArgmaxResult *amax_fine = nullptr;  // refinement argmax (device)
    dg_fix *fix_dev = nullptr;
    dg_fix *fix_host = nullptr;         // pinned
    dg_fix *fix_dev_sync = nullptr, *fix_host_sync = nullptr;  // the same of dg_argmax_refine
    cudaGraphExec_t graph = nullptr;
    int64_t graph_launches = 0;         // kernels per replay
    uint64_t steps_gen = 1, graph_gen = 0;  // capture buffers / formats / lengths generation
    std::string err;
    std::vector<std::shared_ptr<BatchHold>> holds;  // of batches that hold pointers into this context's buffers
    std::vector<void *> retired;        // buffers replaced while a captured step may replay on them (held)
    int64_t launches = 0;
    std::vector<TimedLaunch> pending;
    double ms[DG_K_NCLASS] = {};
    int64_t nl[DG_K_NCLASS] = {};
};

namespace {

dg_status fail(dg_ctx *c, dg_status st, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (c)
        c->err = buf;
    else
        g_thread_error = buf;
    return st;
}

#define CK(ctx, call)                                                                          \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return fail(ctx, e_ == cudaErrorMemoryAllocation ? DG_ENOMEM : DG_ECUDA, "%s: %s", \
                        #call, cudaGetErrorString(e_));                                        \
    } while (0)

size_t iq_bytes(int fmt)
{
    switch (fmt) {
    case DG_IQ_C64: return 8;
    case DG_IQ_CI16: return 4;
    case DG_IQ_CI8: return 2;
    default: return 0;
    }
}

bool finite3(const double *v) { return std::isfinite(v[0]) && std::isfinite(v[1]) && std::isfinite(v[2]); }

// Record kernel timing events around a launch when timing is on.
struct Timed {
    dg_ctx *c;
    int cls;
    cudaEvent_t a = nullptr, b = nullptr;
    Timed(dg_ctx *c_, int cls_) : c(c_), cls(cls_)
    {
        if (c->opt.timing) {
            cudaEventCreate(&a);
            cudaEventCreate(&b);
            cudaEventRecord(a, c->stream);
        }
    }
    void done(int nlaunch)
    {
        c->launches += nlaunch;
        if (c->opt.timing) {
            cudaEventRecord(b, c->stream);
            c->pending.push_back({cls, a, b});
            c->nl[cls] += nlaunch;
            a = b = nullptr;
        }
    }
    ~Timed()
    {
        if (a) cudaEventDestroy(a);
        if (b) cudaEventDestroy(b);
    }
};

dg_status check_latched(dg_ctx *c)
{
    // err_h mirrors err_d after the last enqueued copy; caller has synchronised.
    const unsigned e = *c->err_h;
    if (e) {
        *c->err_h = 0;
        cudaMemsetAsync(c->err_d, 0, sizeof(unsigned), c->stream);
        if (e & ERR_TIMEOUT)
            return fail(c, DG_ETIMEOUT, "a tensor-core pipeline wait ran out of its time budget; the "
                        "affected surface values are not valid");
        if (e & ERR_NU_RANGE)
            return fail(c, DG_EUNSUPPORTED,
                        "a candidate's FDOA exceeds 0.2 fs (|dfreq/fs| > 0.2); the correlation "
                        "kernels do not handle it");
        if (e & ERR_BIN_SPACING)
            return fail(c, DG_EUNSUPPORTED,
                        "CDFT: a snapshot's FDOA span is too wide for its chunk (chunk x bin spacing > 4e-2 "
                        "cycles); use a shorter chunk or DIRECT");
        return fail(c, DG_EUNSUPPORTED, "a candidate's lag |D| exceeds 1e9 samples");
    }
    return DG_OK;
}

// Whether a captured step may still read this context's buffers: its own graph while
// it can be launched (its replays lie before what is freed on the stream), a batch
// while it can be launched or runs on its own stream.
static bool held(dg_ctx *c)
{
    auto runs = [](const BatchHold &h) {
        const bool busy = cudaEventQuery(h.last) != cudaSuccess;
        if (busy) cudaGetLastError();  // not an error of the next launch's
        return busy;
    };
    for (size_t i = 0; i < c->holds.size();) {
        const BatchHold &h = *c->holds[i];
        if (!h.alive || (h.gen != c->steps_gen && !runs(h))) {
            c->holds[i] = c->holds.back();
            c->holds.pop_back();
        } else {
            ++i;
        }
    }
    return !c->holds.empty() || (c->graph && c->graph_gen == c->steps_gen);
}

// The buffers that were kept for captured steps, once no such step is left.
static dg_status give_back(dg_ctx *c)
{
    if ((c->retired.empty() && c->cd.kept.empty()) || held(c)) return DG_OK;
    for (void *p : c->retired) CK(c, cudaFreeAsync(p, c->stream));
    c->retired.clear();
    for (const CdftLayout &L : c->cd.kept)
        for (int *p : {L.bbase, L.gbase})
            if (p) CK(c, cudaFreeAsync(p, c->stream));
    c->cd.kept.clear();
    return DG_OK;
}

// Give a buffer back, or keep it while a captured step may still replay on it.
dg_status release(dg_ctx *c, void *p)
{
    const dg_status st = give_back(c);
    if (st != DG_OK || !p) return st;
    if (held(c)) {
        c->retired.push_back(p);
        return DG_OK;
    }
    CK(c, cudaFreeAsync(p, c->stream));
    return DG_OK;
}

// Make room for another layout in L: the old one is kept where a captured step may
// read its tables, one of the shape asked for comes back (then true): a program
// that alternates between refinement windows holds one layout of each.
static bool swap_layout(dg_ctx *c, CdftLayout &L, int64_t G, int nseg, double diam, bool direct)
{
    auto fits = [&](const CdftLayout &k) {
        if (k.G != G || k.nseg != nseg || k.diam < diam || k.direct != direct || k.batches.empty()) return false;
        for (size_t i = 0; i < k.fmts.size(); ++i)
            if (k.fmts[i] != c->steps[i].fmt) return false;
        return true;
    };
    if (fits(L)) return true;
    if (L.G >= 0 && L.bbase && held(c)) {
        c->cd.kept.push_back(L);
        L = CdftLayout{};
    }
    for (auto k = c->cd.kept.begin(); k != c->cd.kept.end(); ++k) {
        if (!fits(*k)) continue;
        int *const old[2] = {L.bbase, L.gbase};
        L = *k;
        c->cd.kept.erase(k);
        for (int *p : old)
            if (p && release(c, p) != DG_OK) break;
        return true;
    }
    return false;
}

// Device and pinned host memory. A failed call leaves *p NULL, and no error for
// the next launch's cudaGetLastError to find.
template <typename P> cudaError_t device_alloc(dg_ctx *c, P **p, size_t bytes)
{
    const cudaError_t e = cudaMallocAsync((void **)p, bytes, c->stream);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
    }
    return e;
}
template <typename P> cudaError_t pinned_alloc(P **p, size_t bytes)
{
    const cudaError_t e = cudaMallocHost((void **)p, bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
    }
    return e;
}

// At least `bytes` at *p. key (optional): what the buffer holds; 0 once it is
// replaced, so that a failure here or later leaves no description of what is gone.
dg_status ensure(dg_ctx *c, void **p, size_t *cap, size_t bytes, int *key = nullptr)
{
    if (*cap >= bytes && *p) return DG_OK;
    if (key) *key = 0;
    *cap = 0;
    const dg_status st = release(c, *p);
    *p = nullptr;
    if (st != DG_OK) return st;
    CK(c, device_alloc(c, p, bytes));
    *cap = bytes;
    return DG_OK;
}

dg_status push_steps(dg_ctx *c)
{
    if (!c->steps_dirty) return DG_OK;
    for (int k = 0; k < c->K; ++k) {
        c->steps_h[k].y1 = c->steps[k].y1;
        c->steps_h[k].y2 = c->steps[k].y2;
        c->steps_h[k].n = (int)c->steps[k].n;
        c->steps_h[k].fmt = c->steps[k].fmt;
    }
    CK(c, cudaMemcpyAsync(c->steps_d, c->steps_h.data(), sizeof(StepDesc) * c->K,
                          cudaMemcpyHostToDevice, c->stream));
    // steps_h must stay unchanged until that copy has run: it is only
    // rewritten by a later push, which first synchronises.
    CK(c, cudaStreamSynchronize(c->stream));
    c->steps_dirty = false;
    return DG_OK;
}

// Correlation for all snapshots over grid gd (ECEF xyz) into surf [K][G],
// then the ordered sum into out.
// Poll limit of the tensor-core pipeline's waits in every CDFT surface
// launched from now on (0 = the kernels' default); set by
// dg_debug_tc_wait_limit, for tests of the timeout path.
static std::atomic<unsigned> g_tc_wait_polls{0};

dg_status run_surface_cdft(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *surf, void *out,
                           bool refine);
static dg_status map_plan(dg_ctx *c);
static dg_status run_surface_map(dg_ctx *c, void *out);
static dg_status run_surface_lag(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *surf, void *out,
                                 bool refine, bool *done);
// A dg_set_grid that found no memory leaves the context without nodes.
static dg_status need_nodes(dg_ctx *c)
{
    return c->xyz ? DG_OK : fail(c, DG_ENOMEM, "no memory was left for the grid's nodes: set a grid first");
}
static dg_status refine_map(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *out, bool *done,
                            const GridDev *mains, int nmains);

// Surfaces whose candidates look their correlations up in delay-Doppler maps
// (dg_map.cu) instead of the per-lag DFT rows of the contraction: the main
// grid of a context that leaves the launch shape to the library (chunk 0,
// DG_TILES_AUTO) with an arithmetic that is FP32 or claims its accuracy (the
// split forms). The single 16-bit forms keep the tensor-core products the
// caller asked for.
static bool map_options(const dg_ctx *c)
{
    return c->opt.algo == DG_ALGO_CDFT && c->opt.chunk == 0 && c->opt.tiles == DG_TILES_AUTO &&
           c->opt.contract != DG_CONTRACT_BF16 && c->opt.contract != DG_CONTRACT_FP16;
}
static bool map_eligible(const dg_ctx *c) { return map_options(c) && c->G >= kMapMinNodes; }

dg_status run_surface(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *surf, void *out,
                      bool refine)
{
    dg_status st = need_nodes(c);
    if (st != DG_OK) return st;
    if (!refine && map_eligible(c)) {
        if ((st = map_plan(c)) != DG_OK) return st;
        if (c->mp.ok) return run_surface_map(c, out);
    }
    if (refine && map_options(c)) {
        bool done = false;
        if ((st = refine_map(c, gd, xyz, G, out, &done, &c->gd, 1)) != DG_OK || done) return st;
    }
    if (c->opt.algo == DG_ALGO_CDFT) return run_surface_cdft(c, gd, xyz, G, surf, out, refine);
    if (c->opt.prec == DG_PREC_FP32 && c->opt.delay == DG_DELAY_INTEGER) {
        bool done = false;
        if ((st = run_surface_lag(c, gd, xyz, G, surf, out, refine, &done)) != DG_OK || done) return st;
    }
    st = push_steps(c);
    if (st != DG_OK) return st;
    bool same_fmt = true;
    for (int k = 1; k < c->K; ++k) same_fmt &= c->steps[k].fmt == c->steps[0].fmt;
    CorrArgs a{};
    a.xyz = xyz;
    a.eph = c->eph;
    a.steps = c->steps_d;
    a.surf = surf;
    a.err = c->err_d;
    a.nrows = gd.nrows;
    a.nlon = gd.nlon;
    a.G = G;
    a.fs = c->fs;
    a.lambda = c->lambda;
    a.delay = c->opt.delay;
    a.acc = c->opt.acc;
    a.prec = c->opt.prec;
    a.rows = c->opt.rows;
    const size_t esz = c->opt.prec == DG_PREC_FP64 ? 8 : 4;
    {
        Timed t(c, refine ? DG_K_REFINE : DG_K_CORR);
        if (same_fmt) {
            a.K = c->K;
            a.fmt = c->steps[0].fmt;
            CK(c, launch_corr_direct(a, c->stream));
            t.done(1);
        } else {
            for (int k = 0; k < c->K; ++k) {
                CorrArgs b = a;
                b.K = 1;
                b.fmt = c->steps[k].fmt;
                b.eph = c->eph + 12 * (size_t)k;
                b.steps = c->steps_d + k;
                b.surf = (char *)surf + esz * (size_t)G * k;
                CK(c, launch_corr_direct(b, c->stream));
            }
            t.done(c->K);
        }
    }
    {
        Timed t(c, refine ? DG_K_REFINE : DG_K_ACCUM);
        CK(c, launch_accumulate(surf, c->K, G, c->opt.prec, out, c->stream));
        t.done(1);
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    return DG_OK;
}


// n elements in place of what *p holds. Capacities that describe *p are 0 while it
// is replaced (the caller's, set again once all of its buffers are there).
template <typename P>
dg_status grow(dg_ctx *c, P **p, size_t n)
{
    const dg_status st = release(c, *p);
    *p = nullptr;
    if (st != DG_OK) return st;
    CK(c, device_alloc(c, p, sizeof(P) * (n ? n : 1)));
    return DG_OK;
}


// ---------------------------------------------------------------------------
// Host-side planning for the chunked-DFT surface. Nothing here reads device
// results: every size is an upper bound known from the grid and the
// ephemerides, so the device work of a surface is one stream of launches with
// no host synchronisation (and can be captured in a CUDA graph).
// ---------------------------------------------------------------------------

// Lag slots of snapshot k over a grid of diameter diam (metres). By the
// triangle inequality |rho2 - rho1| <= |p2 - p1|, so |D| <= |p2 - p1| fs / c;
// and each range moves by at most the displacement of the candidate, so D
// varies by at most 2 diam fs / c over the grid. Eq. 9 then gives at most
// 2 ceil(bound) + 1 lags; 2 more absorb rounding, and 3 more the stencil of
// the Lagrange4 delay (lags L - 1 .. L + 2 around floor(D)).
static int lag_slots(const dg_ephem &e, double fs, double diam)
{
    const double dx = e.p2[0] - e.p1[0], dy = e.p2[1] - e.p1[1], dz = e.p2[2] - e.p1[2];
    const double span = std::min(2.0 * std::sqrt(dx * dx + dy * dy + dz * dz), 2.0 * diam) * fs / kC;
    return (int)std::min(std::ceil(span), 1.0e9) + 6;
}

// FP64 WGS-84 node position on the host (planning only).
static void host_node_ecef(const GridDev &g, double i, double j, double p[3])
{
    const double e2 = kF * (2.0 - kF);
    const double s0 = std::sin(g.lat0_rad), w = std::sqrt(1.0 - e2 * s0 * s0);
    const double mr = kA * (1.0 - e2) / (w * w * w), nr = kA / w;
    const double lat = g.lat0_rad + (i - 0.5 * (g.nlat - 1)) * (g.dlat_m / mr);
    const double lon = g.lon0_rad + (j - 0.5 * (g.nlon - 1)) * (g.dlon_m / (nr * std::cos(g.lat0_rad)));
    const double sl = std::sin(lat), n = kA / std::sqrt(1.0 - e2 * sl * sl);
    p[0] = n * std::cos(lat) * std::cos(lon);
    p[1] = n * std::cos(lat) * std::sin(lon);
    p[2] = n * (1.0 - e2) * sl;
}

// Diameter bound of the shard: the largest distance between its corners and
// edge midpoints (the grid is a lat/lon rectangle), with a 10 % margin.
static double grid_diameter(const GridDev &g)
{
    double p[9][3];
    int n = 0;
    const double r0 = g.row0, r1 = g.row0 + g.nrows - 1, c1 = g.nlon - 1;
    const double is[3] = {r0, std::round(0.5 * (r0 + r1)), r1}, js[3] = {0.0, std::round(0.5 * c1), c1};
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) host_node_ecef(g, is[a], js[b], p[n++]);
    double d = 0.0;
    for (int a = 0; a < n; ++a)
        for (int b = a + 1; b < n; ++b)
            d = std::max(d, std::sqrt((p[a][0] - p[b][0]) * (p[a][0] - p[b][0]) + (p[a][1] - p[b][1]) * (p[a][1] - p[b][1]) +
                                      (p[a][2] - p[b][2]) * (p[a][2] - p[b][2])));
    return 1.1 * d + 1.0;
}

// The diameter behind the lag slots of a direct surface over `shape`, the context's grid
// or a refinement of it centred on any of its nodes: any two nodes' where the rows
// come within 10 degrees of a pole, the longitudes go around half of the Earth or the
// refinement is wide (there three rows and columns, or another centre's, bound
// nothing; the slots then follow from the receivers' separation).
static double direct_diameter(const dg_ctx *c, const GridDev &shape, bool refine)
{
    const GridDev &g = c->gd;
    const double half = 0.5 * g.nlat * g.dlat_m / 6.33e6, ref = refine ? 0.5 * shape.nlat * shape.dlat_m / 6.33e6 : 0.0;
    const double lon = shape.nlon * shape.dlon_m / (6.33e6 * std::cos(refine ? 1.39 : g.lat0_rad));
    if (std::fabs(g.lat0_rad) + half + ref > 1.39 || ref > 0.02 || lon > 3.0) return 2.0 * kA;
    return grid_diameter(shape);
}

// Curvature bounds of D (samples) and the FDOA (cycles per sample) at
// distances >= rho from receivers `sep` apart with speeds <= v and relative
// motion dv. Over a lattice cell a field stays within half its second
// derivative times the squared half diagonal h of its bilinear interpolant,
// and so of the cell's corner values. Order m of a range's Taylor series is at
// most (2m - 3)!! / rho^(m-1); over the receivers' separation the second
// derivatives of D then differ by at most 3 sep / rho^2 and those of u . v (a
// third derivative of the range) by 15 v sep / rho^3 + 3 dv / rho^2. The
// lattice's own curvature (the parallels' up to 80 degrees, 6 / Earth radius)
// adds that much of the gradients, sep / rho and 3 v sep / rho^2 + dv / rho.
struct Curvature {
    double d, nu;
};
static Curvature field_curvature(const dg_ctx *c, double rho, double sep, double v, double dv)
{
    constexpr double kLattice = 6.0 / 6.3e6;
    const double d2 = 3.0 * sep / (rho * rho) + kLattice * sep / rho;
    const double n2 = 15.0 * v * sep / (rho * rho * rho) + 3.0 * dv / (rho * rho) +
                      kLattice * (3.0 * v * sep / (rho * rho) + dv / rho);
    return {d2 * c->fs / kC, n2 / (c->lambda * c->fs)};
}

// Longitudes of a grid's columns, from the first to the last (radians, a little more).
static double lon_extent(const GridDev &g) { return g.nlon * g.dlon_m / (6.33e6 * std::cos(g.lat0_rad)); }

// FDOA span of every snapshot over the shard, from a lattice of nodes (its
// corners, edges and interior; the FDOA field is smooth at these scales): up
// to 65 x 65 nodes, fewer on small shards (at least 9 x 9, about one lattice
// node per 8 grid nodes), the node positions computed once for all
// snapshots. lags: the lattice's lag counts. range: bounds of D and the FDOA
// that hold at every node of the shard (range_bounds).
static void fdoa_spans(const dg_ctx *c, const GridDev &g, std::vector<double> &span,
                       std::vector<double> *lags = nullptr, std::vector<GridRange> *range = nullptr)
{
    const int side = std::max(g.nrows, g.nlon);
    const int lattice = std::min(65, std::max(9, side / 8 + 1));
    const int ni = std::min(lattice, g.nrows), nj = std::min(lattice, g.nlon);
    std::vector<double> p(3 * (size_t)ni * nj);
    for (int a = 0; a < ni; ++a)
        for (int b = 0; b < nj; ++b) {
            const double i = g.row0 + (ni > 1 ? (double)a * (g.nrows - 1) / (ni - 1) : 0.0);
            const double j = nj > 1 ? (double)b * (g.nlon - 1) / (nj - 1) : 0.0;
            host_node_ecef(g, std::round(i), std::round(j), &p[3 * ((size_t)a * nj + b)]);
        }
    double h = 0.0;  // half the longest cell diagonal, with 5 % for the curvature within a cell
    // within 80 degrees, and at most once around: lattice nodes whole turns apart bound nothing
    const bool low = std::fabs(g.lat0_rad) + 0.5 * g.nlat * g.dlat_m / 6.33e6 < 1.39 && lon_extent(g) < 2.0 * kPi;
    if (range) {
        auto dist2 = [&](size_t q, size_t r) {
            const double *x = &p[3 * q], *y = &p[3 * r];
            return (x[0] - y[0]) * (x[0] - y[0]) + (x[1] - y[1]) * (x[1] - y[1]) + (x[2] - y[2]) * (x[2] - y[2]);
        };
        double hi = 0.0, hj = 0.0;
        for (int a = 0; a < ni; ++a)
            for (int b = 0; b < nj; ++b) {
                const size_t q = (size_t)a * nj + b;
                if (a + 1 < ni) hi = std::max(hi, dist2(q, q + nj));
                if (b + 1 < nj) hj = std::max(hj, dist2(q, q + 1));
            }
        h = 0.5 * 1.05 * std::sqrt(hi + hj);
        GridRange R0{};  // the steps, with 2 % for their change within a cell
        R0.row_m = ni > 1 ? 1.02 * std::sqrt(hi) / std::floor((double)(g.nrows - 1) / (ni - 1)) : 0.0;
        R0.col_m = nj > 1 ? 1.02 * std::sqrt(hj) / std::floor((double)(g.nlon - 1) / (nj - 1)) : 0.0;
        range->assign(c->K, R0);
    }
    span.assign(c->K, 0.0);
    if (lags) lags->assign(c->K, 1.0);
    for (int k = 0; k < c->K; ++k) {
        double lo = 1e300, hi = -1e300, dlo = 1e300, dhi = -1e300, rmin = 1e300;
        const dg_ephem &e = c->eph_host[k];
        for (size_t q = 0; q < (size_t)ni * nj; ++q) {
            const double *x = &p[3 * q];
            double f[2], r[2];  // Eq. 6-8 and 4, 7
            for (int t = 0; t < 2; ++t) {
                const double *pp = t ? e.p2 : e.p1, *vv = t ? e.v2 : e.v1;
                const double dx = pp[0] - x[0], dy = pp[1] - x[1], dz = pp[2] - x[2];
                r[t] = std::sqrt(dx * dx + dy * dy + dz * dz);
                f[t] = -(dx * vv[0] + dy * vv[1] + dz * vv[2]) / (r[t] * c->lambda);
            }
            const double nu = f[1] - f[0];  // times fs
            lo = std::min(lo, nu);
            hi = std::max(hi, nu);
            if (lags) {  // Eq. 7 and 9: the lattice's lag range
                const double D = (r[1] - r[0]) * c->fs / kC;
                dlo = std::min(dlo, D);
                dhi = std::max(dhi, D);
                rmin = std::min(rmin, std::min(r[0], r[1]));
            }
        }
        lo /= c->fs;
        hi /= c->fs;
        span[k] = hi - lo;
        if (lags) (*lags)[k] = std::floor(dhi + 0.5) - std::floor(dlo + 0.5) + 1.0;
        if (lags && range) {
            auto norm = [](double x, double y, double z) { return std::sqrt(x * x + y * y + z * z); };
            const double sep = norm(e.p2[0] - e.p1[0], e.p2[1] - e.p1[1], e.p2[2] - e.p1[2]);
            const double dv = norm(e.v2[0] - e.v1[0], e.v2[1] - e.v1[1], e.v2[2] - e.v1[2]);
            const double v = std::max(norm(e.v1[0], e.v1[1], e.v1[2]), norm(e.v2[0], e.v2[1], e.v2[2]));
            const double rho = rmin - h - 0.5 * sep;  // also along the receivers' segment
            GridRange &R = (*range)[k];
            if (rho > 0.0 && low) {
                const Curvature q = field_curvature(c, rho, sep, v, dv);
                const double md = 0.5 * q.d * h * h, mn = 0.5 * q.nu * h * h;
                R.d_lo = dlo - md;
                R.d_hi = dhi + md;
                R.nu_lo = lo - mn;
                R.nu_hi = hi + mn;
                R.rho = rho;
            } else {
                R.d_lo = R.nu_lo = -1e300;
                R.d_hi = R.nu_hi = 1e300;
            }
            R.sep = sep;
            R.vel = v;
        }
    }
}

// Chunk of a batch with chunk = 0: the longest power of two in
// [64, kCdftAutoMaxChunk] (tensor cores: [64, kCdftAutoMaxChunkTc]) whose
// length times the estimated bin spacing stays within kCdftMDelta / 1.1 (a
// margin for the lattice estimate; the plan kernel checks the bound against
// the exact spacing). On the tensor cores a chunk above kCdftAutoMaxChunk is
// kept only while it fits every capture of the batch and the batch still
// has kCdftMinTilesPerSm lag tiles (128 lags x one chunk, from the lattice's
// lag counts) per SM: longer chunks mean fewer per-lag DFT rows to write and
// to merge into super-chunks, but fewer and longer tiles.
static int auto_chunk(const dg_ctx *c, const std::vector<double> &span, const std::vector<double> &lags, int k0,
                      int S, bool tc)
{
    double dmax = 0.0;
    int64_t nmin = INT64_MAX;
    for (int s = 0; s < S; ++s) {
        dmax = std::max(dmax, span[k0 + s] * (1.0 + 1e-5) / kCdftBinSpan);
        nmin = std::min<int64_t>(nmin, c->steps[k0 + s].n);
    }
    int M = tc ? kCdftAutoMaxChunkTc : kCdftAutoMaxChunk;
    while (M > 64 && 1.1 * M * dmax > kCdftMDelta) M >>= 1;
    auto tiles = [&](int m) {
        double t = 0.0;
        for (int s = 0; s < S; ++s)
            t += std::ceil((double)c->steps[k0 + s].n / m) * std::ceil(lags[k0 + s] / 128.0);
        return t;
    };
    while (M > kCdftAutoMaxChunk && (M > nmin || tiles(M) < (double)kCdftMinTilesPerSm * c->sm_count)) M >>= 1;
    return M;
}

// The batches of snapshots of a surface of G nodes (same IQ format, scratch
// within the context's target) and their bucket / combine-group bases.
// Snapshots per batch: per-candidate arrays (16 B per candidate) and the
// per-lag DFTs (lag slots x chunks x 512 B, chunks at the longest automatic
// chunk unless one is fixed) within the scratch target.
static dg_status cdft_batches(dg_ctx *c, int64_t G, double diam, CdftLayout &L, std::vector<int> &bb,
                              std::vector<int> &gb)
{
    const double budget = (double)(c->opt.scratch_mib ? c->opt.scratch_mib : 12288) * 1048576.0;
    int64_t nmax = 1;
    int slots_max = 1;
    for (int k = 0; k < c->K; ++k) {
        nmax = std::max<int64_t>(nmax, c->steps[k].n);
        slots_max = std::max(slots_max, lag_slots(c->eph_host[k], c->fs, diam));
    }
    const int m_est = c->opt.chunk ? c->opt.chunk : kCdftAutoMaxChunk;
    const double per_snap = 16.0 * (double)G + (double)slots_max * (double)((nmax + m_est - 1) / m_est) * 512.0;
    int s_max = (int)std::max<int64_t>(1, std::min<int64_t>(c->K, (int64_t)(budget / per_snap)));
    if (c->opt.contract != DG_CONTRACT_FP32) s_max = std::min(s_max, kTcMaxSnapshots);
    for (int k0 = 0; k0 < c->K;) {
        int S = 1;  // same format, at most s_max snapshots
        while (k0 + S < c->K && S < s_max && c->steps[k0 + S].fmt == c->steps[k0].fmt) ++S;
        CdftLayout::Batch t{k0, S, (int)bb.size(), 0, 0};
        int64_t nb = 0, ng = 0;
        for (int s = 0; s <= S; ++s) {
            bb.push_back((int)nb);
            gb.push_back((int)ng);
            if (s == S) break;
            const int slots = lag_slots(c->eph_host[k0 + s], c->fs, diam);
            nb += slots;
            ng += G / kCdftCombineGroup + slots + 1;
        }
        if (nb > INT_MAX / 64 || ng > INT_MAX)
            return fail(c, DG_EUNSUPPORTED, "CDFT: %lld lag slots in one batch; use DIRECT", (long long)nb);
        t.nbt = nb;
        t.groups = ng;
        L.batches.push_back(t);
        L.s_max = std::max(L.s_max, S);
        L.nbt_max = std::max<int64_t>(L.nbt_max, nb);
        L.groups_max = std::max<int64_t>(L.groups_max, ng);
        k0 += S;
    }
    return DG_OK;
}

// The batches of a surface and their bucket / combine-group bases: static for
// a grid size G (the main grid and the refinement grid each keep one).
static dg_status cdft_layout(dg_ctx *c, const GridDev &gd, int64_t G, CdftLayout &L)
{
    const double diam = grid_diameter(gd);
    if (swap_layout(c, L, G, 0, diam, false)) return DG_OK;
    int *old_bb = L.bbase, *old_gb = L.gbase;
    L = CdftLayout{};
    L.diam = diam;
    for (const Step &t : c->steps) L.fmts.push_back(t.fmt);
    L.bbase = old_bb;
    L.gbase = old_gb;
    std::vector<int> bb, gb;
    dg_status bst = cdft_batches(c, G, diam, L, bb, gb);
    if (bst != DG_OK) return bst;
    dg_status st;
    if ((st = grow(c, &L.bbase, bb.size())) != DG_OK) return st;
    if ((st = grow(c, &L.gbase, gb.size())) != DG_OK) return st;
    // pageable sources: staged before the calls return
    CK(c, cudaMemcpyAsync(L.bbase, bb.data(), sizeof(int) * bb.size(), cudaMemcpyHostToDevice, c->stream));
    CK(c, cudaMemcpyAsync(L.gbase, gb.data(), sizeof(int) * gb.size(), cudaMemcpyHostToDevice, c->stream));
    L.G = G;  // its tables are in place
    return DG_OK;
}

// Chunked-DFT surface. Per batch of snapshots (same IQ format, scratch
// within the context's target): geometry, plan (sort by lag
// bucket and bin, bins, tiles), DFT tables, contraction, super-chunks,
// combine. Then the ordered sum. No host synchronisation.
// The ephemerides as double-float (hi, lo) pairs on the device, [K][24].
static dg_status ensure_ephf(dg_ctx *c)
{
    CdftBufs &b = c->cd;
    if (b.ephf_cap >= (size_t)c->K) return DG_OK;
    dg_status st;
    if ((st = grow(c, &b.ephf, 24 * (size_t)c->K)) != DG_OK) return st;
    std::vector<float> ef(24 * (size_t)c->K);
    for (int k = 0; k < c->K; ++k) {
        const double *v = &c->eph_host[k].p1[0];
        for (int t = 0; t < 12; ++t) {
            ef[24 * k + 2 * t] = (float)v[t];
            ef[24 * k + 2 * t + 1] = (float)(v[t] - (double)ef[24 * k + 2 * t]);
        }
    }
    // pageable source: staged before the call returns
    CK(c, cudaMemcpyAsync(b.ephf, ef.data(), sizeof(float) * ef.size(), cudaMemcpyHostToDevice, c->stream));
    b.ephf_cap = (size_t)c->K;
    return DG_OK;
}

// The nodes' double-float split, G of them.
static dg_status ensure_xyzf(dg_ctx *c, int64_t G)
{
    CdftBufs &b = c->cd;
    return ensure(c, (void **)&b.xyzf, &b.xyzf_cap, sizeof(float) * 6 * (size_t)G);
}

// Scratch of the lag sort, grown on demand (never inside a captured graph: a
// graph is captured after one uncaptured call of the same shape): S snapshots,
// SG (snapshot, candidate) pairs, nbt lag slots, groups combine groups.
static dg_status ensure_sort(dg_ctx *c, size_t S, size_t SG, size_t nbt, size_t groups)
{
    CdftBufs &b = c->cd;
    dg_status st;
    if (b.s_cap < S) {
        b.s_cap = 0;
        if ((st = grow(c, &b.lr, 2 * S)) != DG_OK) return st;
        if ((st = grow(c, &b.delta, S)) != DG_OK) return st;
        if ((st = grow(c, &b.nubase, S)) != DG_OK) return st;
        if ((st = grow(c, &b.nur, 2 * S)) != DG_OK) return st;
        if ((st = grow(c, &b.tbase, S + 1)) != DG_OK) return st;
        if ((st = grow(c, &b.hbase, S + 1)) != DG_OK) return st;
        if ((st = grow(c, &b.layout, S)) != DG_OK) return st;
        if ((st = grow(c, &b.Mcs, S)) != DG_OK) return st;
        b.s_cap = S;
    }
    if (b.sg_cap < SG) {
        b.sg_cap = 0;
        if ((st = grow(c, &b.candL, SG)) != DG_OK) return st;
        if ((st = grow(c, &b.candNu, SG)) != DG_OK) return st;
        if ((st = grow(c, &b.order, SG)) != DG_OK) return st;
        if ((st = grow(c, &b.nuS, SG)) != DG_OK) return st;
        b.sg_cap = SG;
    }
    if (b.nb_cap < nbt) {
        b.nb_cap = 0;
        if ((st = grow(c, &b.count, nbt)) != DG_OK) return st;
        if ((st = grow(c, &b.need, nbt)) != DG_OK) return st;
        if ((st = grow(c, &b.offs, nbt)) != DG_OK) return st;
        if ((st = grow(c, &b.subcnt, nbt)) != DG_OK) return st;
        b.nb_cap = nbt;
    }
    if (b.g2b_cap < groups) {
        b.g2b_cap = 0;
        if ((st = grow(c, &b.g2b, groups)) != DG_OK) return st;
        b.g2b_cap = groups;
    }
    return DG_OK;
}

// The arguments of the geometry and the lag sort of one batch.
static void sort_args(dg_ctx *c, const CdftLayout::Batch &bt, const CdftLayout &L, const GridDev &gd, const double *xyz,
                      int64_t G, CdftBatch &a)
{
    CdftBufs &b = c->cd;
    auto split = [](double d, float &h, float &l) {  // constants as double-float (hi, lo) pairs
        h = (float)d;
        l = (float)(d - (double)h);
    };
    a.xyz = xyz;
    a.xyzf = b.xyzf;
    a.ephf = b.ephf + 24 * (size_t)bt.k0;
    split(c->fs / kC, a.fsc_hi, a.fsc_lo);
    split(1.0 / (c->lambda * c->fs), a.ilf_hi, a.ilf_lo);
    a.eph = c->eph + 12 * (size_t)bt.k0;
    a.sd = c->steps_d + bt.k0;
    a.S = bt.S;
    a.k0 = bt.k0;
    a.G = G;
    a.nrows = gd.nrows;
    a.nlon = gd.nlon;
    a.fs = c->fs;
    a.lambda = c->lambda;
    a.acc = c->opt.acc;
    a.err = c->err_d;
    a.lr = b.lr;
    a.nur = b.nur;
    a.nubase = b.nubase;
    a.delta = b.delta;
    a.bbase = L.bbase + bt.base;
    a.gbase = L.gbase + bt.base;
    a.candL = b.candL;
    a.candNu = b.candNu;
    a.order = b.order;
    a.nuS = b.nuS;
    a.g2b = b.g2b;
    a.count = b.count;
    a.need = b.need;
    a.offs = b.offs;
    a.subcnt = b.subcnt;
    a.delay = c->opt.delay;
    a.candMu = b.candMu;
    a.muS = b.muS;
    a.ngroups = (int)bt.groups;
}

// Tiles per SM of a whole grid and all snapshots (k_corr_direct at 8 rows a thread).
static double grid_tiles(const dg_ctx *c, const GridDev &g)
{
    return std::ceil(g.nlat / 64.0) * std::ceil(g.nlon / 32.0) * c->K / c->sm_count;
}

// Whether the tile kernel (k_corr_direct) is the faster one for an FP32 surface
// with integer delays: where few candidates share a lag. k_corr_lag takes a warp
// per group however few candidates it has, 5.1e-6 us per group and sample on 152
// SMs; the tile kernel takes a CTA per rows x 256 candidates, on widely spread lags
// 0.145 us per tile of an SM and sample plus 0.1, 0.36 at least (tiles of 8 rows,
// whatever dg_options.rows asks for: a surface is the same bits for every value;
// lower envelopes of what it took, so that no grid is slower than on its tiles).
// Measured, grouped against tiles, by candidates per group: 401^2 nodes and 16
// snapshots of 16384 samples 7.2 against 19.0 ms (46), 10.7 / 26.2 (25), 24.8 / 26.0
// (8.6), 29.2 / 26.4 (7.3), 51.6 / 33.1 (4.1), 125 / 37.8 (1.7); 201^2 and 8 of 32768
// 13.1 / 14.3 (4.1), 18.2 / 21.6 (3.0), 20.5 / 15.5 (2.6), 36.7 / 17.5 (1.5); 101^2 and
// 8 of 32768, which leave most SMs without a tile, 12.1 / 12.7 (1.2).
// The groups are estimated from the lags at a lattice of 9 x 9 nodes (0.88 of what an
// even spread over their range would give, as counted on those grids) of the
// whole grid, so that every row shard of it takes the same kernel. A refinement
// grid (gd) is judged as if on the main grid's centre. In a batch the other
// contexts' work fills the SMs that a small grid's tiles leave: a context's tiles
// then cost their share of the whole batch's (32 contexts of 101^2 nodes, 4
// snapshots of 16384 samples: 10.2 / 15.7 ms at 15 candidates a group, 33.7 / 22.9 at
// 3.6, 48.0 / 21.3 at 2.5), and its synchronising calls go the same way while the
// batch can be launched.
static bool tiles_faster(const dg_ctx *c, const GridDev &gd, LagRule &rule)
{
    GridDev g = gd;
    g.row0 = 0;
    g.nrows = g.nlat;
    const double tiles = grid_tiles(c, g);
    double fill = std::max(tiles, c->cd.fill);
    for (const auto &h : c->holds)
        if (h->alive && h->gen == c->steps_gen) fill = std::max(fill, h->fill);
    const GridDev &o = rule.g;
    if (rule.known && rule.fill == fill && o.lat0_rad == g.lat0_rad && o.lon0_rad == g.lon0_rad && o.dlat_m == g.dlat_m && o.dlon_m == g.dlon_m &&
        o.nlat == g.nlat && o.nlon == g.nlon)
        return rule.tiles;
    const int ni = std::min(9, g.nlat), nj = std::min(9, g.nlon);
    std::vector<double> p(3 * (size_t)ni * nj);
    for (int i = 0; i < ni; ++i)
        for (int j = 0; j < nj; ++j)
            host_node_ecef(g, ni > 1 ? (double)i * (g.nlat - 1) / (ni - 1) : 0.0, nj > 1 ? (double)j * (g.nlon - 1) / (nj - 1) : 0.0,
                           &p[3 * ((size_t)i * nj + j)]);
    const double G = (double)g.nlat * g.nlon;
    double groups = 0.0;
    for (int k = 0; k < c->K; ++k) {
        const dg_ephem &e = c->eph_host[k];
        double lo = 1e300, hi = -1e300;
        for (size_t q = 0; q < p.size(); q += 3) {
            const double *x = &p[q];
            double r[2];
            for (int t = 0; t < 2; ++t) {
                const double *s = t ? e.p2 : e.p1;
                r[t] = std::sqrt((s[0] - x[0]) * (s[0] - x[0]) + (s[1] - x[1]) * (s[1] - x[1]) + (s[2] - x[2]) * (s[2] - x[2]));
            }
            lo = std::min(lo, r[1] - r[0]);
            hi = std::max(hi, r[1] - r[0]);
        }
        const double lags = (hi - lo) * c->fs / kC + 1.0;
        groups += 0.88 * (lags * -std::expm1(-G / lags) + G / kDirectGroup);  // the lags that hold a candidate
    }
    rule.g = g;
    rule.fill = fill;
    rule.known = true;
    rule.tiles = groups * 5.1e-6 * 152.0 / c->sm_count > std::max(0.36, 0.1 + 0.145 * fill) * tiles / fill;
    return rule.tiles;
}

// The batches of snapshots of a grouped surface, their lag tables, and the buffers of
// its sort, within the scratch target: 24 bytes a node, and per snapshot (4 GiB at
// most) 16 a node, a lag slot and a group, and 8 a node and segment of samples.
// *fits = false where one snapshot needs more.
static dg_status lag_batches(dg_ctx *c, CdftLayout &L, int64_t G, double diam, int nseg, bool *fits)
{
    CdftBufs &b = c->cd;
    dg_status st;
    *fits = false;
    if (!swap_layout(c, L, G, nseg, diam, true)) {
        const double budget = (double)(c->opt.scratch_mib > 0 ? c->opt.scratch_mib : 12288) * 1048576.0;
        CdftLayout n;
        n.G = G;
        n.nseg = nseg;
        n.direct = true;
        n.diam = diam;
        int slots_max = 1;
        for (int k = 0; k < c->K; ++k) slots_max = std::max(slots_max, lag_slots(c->eph_host[k], c->fs, diam));
        const double seg = nseg > 1 ? 8.0 * (double)G * nseg : 0.0;
        const double per = 16.0 * ((double)G + 2.0 * slots_max + (double)G / kDirectGroup + 2.0) + seg;
        const double sorts = std::min(4294967296.0, budget - 24.0 * (double)G);
        const int s_max = (int)std::max(1.0, std::min((double)std::min(c->K, 65535), std::floor(sorts / per)));
        std::vector<int> bb, gb;
        for (int k0 = 0; k0 < c->K; k0 += s_max) {
            const int S = std::min(s_max, c->K - k0);
            CdftLayout::Batch t{k0, S, (int)bb.size(), 0, 0};
            for (int s = 0; s <= S; ++s) {
                if (t.nbt > (1 << 26) || t.groups > (1 << 30)) return DG_OK;
                bb.push_back((int)t.nbt);
                gb.push_back((int)t.groups);
                if (s == S) break;
                const int slots = lag_slots(c->eph_host[k0 + s], c->fs, diam);
                t.nbt += slots;
                t.groups += G / kDirectGroup + slots + 1;
            }
            n.batches.push_back(t);
            n.s_max = std::max(n.s_max, S);
            n.nbt_max = std::max(n.nbt_max, t.nbt);
            n.groups_max = std::max(n.groups_max, t.groups);
        }
        if (24.0 * (double)G + per * n.s_max > budget) return DG_OK;
        n.bbase = L.bbase;
        n.gbase = L.gbase;
        L = n;
        L.G = -1;  // until its tables are in place
        if ((st = grow(c, &L.bbase, bb.size())) != DG_OK) return st;
        if ((st = grow(c, &L.gbase, gb.size())) != DG_OK) return st;
        // pageable sources: staged before the calls return
        CK(c, cudaMemcpyAsync(L.bbase, bb.data(), sizeof(int) * bb.size(), cudaMemcpyHostToDevice, c->stream));
        CK(c, cudaMemcpyAsync(L.gbase, gb.data(), sizeof(int) * gb.size(), cudaMemcpyHostToDevice, c->stream));
        L.G = G;
    }
    const size_t S = (size_t)L.s_max, SG = S * (size_t)G;
    if ((st = ensure_sort(c, S, SG, (size_t)L.nbt_max, (size_t)L.groups_max)) != DG_OK) return st;
    if (nseg > 1 && (st = ensure(c, (void **)&b.part, &b.part_cap, sizeof(float2) * SG * nseg)) != DG_OK) return st;
    if ((st = ensure_ephf(c)) != DG_OK) return st;
    if ((st = ensure_xyzf(c, G)) != DG_OK) return st;
    *fits = true;
    return DG_OK;
}

// The direct FP32 surface with the candidates grouped by lag (k_corr_lag):
// per batch of snapshots (lag_batches) the chunked-DFT path's
// geometry and lag sort, then the correlation. *done = false where the tile kernel
// is the faster one (tiles_faster), where the lag slots or the captures are out of
// its range, and where the sort does not fit the scratch target, or the memory there
// is: then until the shapes change, so that a captured step takes the same route.
static dg_status run_surface_lag(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *surf, void *out,
                                 bool refine, bool *done)
{
    *done = false;
    CdftBufs &b = c->cd;
    CdftLayout &L = refine ? b.dloc_layout : b.dmain_layout;
    for (int k = 0; k < c->K; ++k)
        if (c->steps[k].n > (1 << 24) || !c->steps[k].loaded) return DG_OK;
    if (tiles_faster(c, gd, refine ? b.dloc_rule : b.dmain_rule)) return DG_OK;
    if (b.no_sort == c->steps_gen) return DG_OK;
    // segments of samples: enough warps for about 8 rounds of the chip at 48
    // warps per SM, from the whole grid's size (a row shard sums alike), in
    // multiples of 256 samples
    int nmax = 1;
    for (int k = 0; k < c->K; ++k) nmax = std::max(nmax, (int)c->steps[k].n);
    const double warps = (double)gd.nlat * gd.nlon / 32.0 * c->K;
    const int want = (int)std::min(64.0, std::ceil(8.0 * 48.0 * 152.0 / std::max(warps, 1.0)));
    const int seg_len = std::max(1, (nmax + 256 * want - 1) / (256 * want)) * 256;
    const int nseg = (nmax + seg_len - 1) / seg_len;
    GridDev shape = gd;  // as in cdft_setup: a captured refinement's centre is known on the device only
    if (refine) {
        shape.lat0_rad = c->gd.lat0_rad;
        shape.lon0_rad = c->gd.lon0_rad;
    }
    dg_status st = push_steps(c);
    if (st != DG_OK) return st;
    bool fits = false;
    st = lag_batches(c, L, G, direct_diameter(c, shape, refine), nseg, &fits);
    if (st == DG_ENOMEM) {
        c->err.clear();
        b.no_sort = c->steps_gen;
        return DG_OK;
    }
    if (st != DG_OK || !fits) return st;
    const bool one = L.batches.size() == 1;
    {
        Timed t(c, refine ? DG_K_REFINE : DG_K_CORR);
        CK(c, launch_ecef_split(xyz, G, b.xyzf, c->stream, one ? b.lr : nullptr, b.nur, one ? L.s_max : 0));
        t.done(1);
    }
    int slots = 0;
    for (int k = 0; k < c->K; ++k) slots = std::max(slots, lag_slots(c->eph_host[k], c->fs, L.diam));
    // one CTA sorts a snapshot where that is shorter than the three launches
    const bool small = G <= kSortNodes && slots <= kSortSlots;
    const bool fused = one && nseg > 1;  // the segments' sums go straight into the sum over snapshots
    for (const auto &bt : L.batches) {
        CdftBatch a{};
        sort_args(c, bt, L, gd, xyz, G, a);
        a.group = kDirectGroup;
        a.nu_max = 0.2f;
        a.mma = 1;  // no FP32 DFT table
        a.lr_ready = one;
        Timed t(c, refine ? DG_K_REFINE : DG_K_CORR);
        CK(c, launch_cdft_geo(a, c->stream));
        int n = one ? 1 : 2;
        if (small) {
            CK(c, launch_sort_small(a, c->stream));
            n += 1;
        } else {
            CK(c, cudaMemsetAsync(b.g2b, 0xff, sizeof(int4) * (size_t)bt.groups, c->stream));
            CK(c, launch_cdft_plan(a, (int)bt.nbt, c->stream));
            n += 3;
        }
        float *sf = (float *)surf;
        CK(c, launch_corr_lag(a, nseg, seg_len, sf, nseg > 1 ? b.part : nullptr, c->stream));
        ++n;
        if (nseg > 1) {
            CK(c, launch_corr_segments(b.part, bt.S, nseg, G, c->opt.acc, sf + (size_t)bt.k0 * G,
                                       fused ? (float *)out : nullptr, c->stream));
            ++n;
        }
        t.done(n);
    }
    if (!fused) {
        Timed t(c, refine ? DG_K_REFINE : DG_K_ACCUM);
        CK(c, launch_accumulate(surf, c->K, G, DG_PREC_FP32, out, c->stream));
        t.done(1);
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    *done = true;
    return DG_OK;
}

// The phases of one chunked-DFT surface: setup (layout, chunks, buffers,
// the candidates' double-float split), then per batch of snapshots its
// arguments, plan, contraction and combine, then the ordered accumulation.
// run_surface_cdft runs them in order; a batch of contexts captured as one
// graph (dg_batch_capture) runs the contraction of the r-th batch of every
// context as one persistent launch between the plans and the combines.
static dg_status cdft_setup(dg_ctx *c, CdftRun &r)
{
    const GridDev &gd = r.gd;
    const double *xyz = r.xyz;
    const int64_t G = r.G;
    const bool refine = r.refine;
    dg_status st = push_steps(c);
    if (st != DG_OK) return st;
    for (int k = 0; k < c->K; ++k)
        if (c->steps[k].n > (1 << 24))
            return fail(c, DG_EUNSUPPORTED, "CDFT: snapshots longer than 2^24 samples are not supported; use DIRECT");
    CdftBufs &b = c->cd;
    CdftLayout &L = refine ? b.loc_layout : b.main_layout;
    r.L = &L;
    // a refinement grid is planned from its shape only (as if centred on the
    // main grid's centre), so that a step captured in a CUDA graph, whose
    // refinement centre is known on the device only, plans it alike
    GridDev shape = gd;
    if (refine) {
        shape.lat0_rad = c->gd.lat0_rad;
        shape.lon0_rad = c->gd.lon0_rad;
    }
    if ((st = cdft_layout(c, shape, G, L)) != DG_OK) return st;
    const int s_max = L.s_max;
    // FDOA spans for the automatic chunk, from the main grid (a refinement
    // grid lies around one of its nodes and spans far less)
    std::vector<double> &span = b.main_span;
    const bool mma = c->opt.contract != DG_CONTRACT_FP32;
    r.mma = mma;
    if (c->opt.chunk == 0 && (span.size() != (size_t)c->K || b.main_lags.size() != (size_t)c->K))
        fdoa_spans(c, c->gd, span, &b.main_lags, &b.main_range);
    std::vector<int> &Ms = r.Ms;
    Ms.assign(L.batches.size(), 0);
    int M_max = 64, B_max = 1;
    for (size_t i = 0; i < L.batches.size(); ++i) {
        const auto &t = L.batches[i];
        // Hankel tiles take chunks of at most kLagTileMaxChunk
        const bool tc = mma && c->opt.tiles != DG_TILES_HANKEL;
        Ms[i] = c->opt.chunk ? c->opt.chunk : auto_chunk(c, span, b.main_lags, t.k0, t.S, tc);
        if (refine && !c->opt.chunk) Ms[i] = std::min(Ms[i], kCdftRefineMaxChunk);
        M_max = std::max(M_max, Ms[i]);
        for (int s = 0; s < t.S; ++s) B_max = std::max<int>(B_max, (int)((c->steps[t.k0 + s].n + Ms[i] - 1) / Ms[i]));
    }
    // scratch, grown on demand (never inside a captured graph: a graph is
    // captured after one uncaptured call of the same shape)
    if ((st = ensure_sort(c, (size_t)s_max, (size_t)s_max * G, (size_t)L.nbt_max, (size_t)L.groups_max)) != DG_OK)
        return st;
    if (!b.work) {
        if ((st = grow(c, &b.work, 2)) != DG_OK) return st;
    }
    if (c->opt.delay != DG_DELAY_INTEGER && b.mu_cap < (size_t)s_max * G) {
        b.mu_cap = 0;
        if ((st = grow(c, &b.candMu, (size_t)s_max * G)) != DG_OK) return st;
        if ((st = grow(c, &b.muS, (size_t)s_max * G)) != DG_OK) return st;
        b.mu_cap = (size_t)s_max * G;
    }
    if (!mma && b.v_cap < (size_t)s_max * M_max * 64) {  // the FP32 contraction's DFT table
        b.v_cap = 0;
        if ((st = grow(c, &b.V, (size_t)s_max * M_max * 64)) != DG_OK) return st;
        b.v_cap = (size_t)s_max * M_max * 64;
    }
    const size_t w_elems = (size_t)L.nbt_max * (size_t)B_max * 128;
    if (w_elems * sizeof(float) > ((size_t)64 << 30))
        return fail(c, DG_EUNSUPPORTED, "CDFT: the per-lag DFT buffer would exceed 64 GiB (%lld lag slots x %d chunks); "
                    "use a longer chunk or DIRECT", (long long)L.nbt_max, B_max);
    if (b.w_cap < w_elems) {
        b.w_cap = 0;
        if ((st = grow(c, &b.W, w_elems)) != DG_OK) return st;
        b.w_cap = w_elems;
    }
    if (mma) {
        const size_t bt = (size_t)s_max * cdft_btab_bytes(c->opt.contract, M_max);
        if ((st = ensure(c, &b.btab, &b.btab_cap, bt)) != DG_OK) return st;
    }
    const int kplan = refine ? DG_K_REFINE : DG_K_CDFT_PLAN;
    if (!refine) {
        CK(c, cudaMemsetAsync(b.work, 0, 2 * sizeof(unsigned long long), c->stream));
        c->cd_chunk_min = INT_MAX;
        c->cd_chunk_max = 0;
    }
    if ((st = ensure_ephf(c)) != DG_OK) return st;
    if ((st = ensure_xyzf(c, G)) != DG_OK) return st;
    {
        Timed t(c, kplan);
        CK(c, launch_ecef_split(xyz, G, b.xyzf, c->stream));
        t.done(1);
    }
    if (!refine) c->cd.main_run = r;
    return DG_OK;
}

static void cdft_args(dg_ctx *c, const CdftRun &r, size_t bi, CdftBatch &a)
{
    CdftBufs &b = c->cd;
    const CdftLayout &L = *r.L;
    const std::vector<int> &Ms = r.Ms;
    const bool mma = r.mma, refine = r.refine;
    const double *xyz = r.xyz;
    const GridDev &gd = r.gd;
    const int64_t G = r.G;
    const auto &bt = L.batches[bi];
    const int k0 = bt.k0, S = bt.S, M = Ms[bi];
    int Bmax = 1;
    for (int s = 0; s < S; ++s) Bmax = std::max<int>(Bmax, (int)((c->steps[k0 + s].n + M - 1) / M));
    if (!refine) {
        c->cd_chunk_min = std::min(c->cd_chunk_min, M);
        c->cd_chunk_max = std::max(c->cd_chunk_max, M);
    }
    sort_args(c, bt, L, gd, xyz, G, a);
    a.M = M;
    a.Bmax = Bmax;
    a.V = b.V;
    a.W = b.W;
    a.tbase = b.tbase;
    a.hbase = b.hbase;
    a.layout = b.layout;
    a.Mcs = b.Mcs;
    a.work = refine ? nullptr : b.work;
    a.group = kCdftCombineGroup;
    a.tiles_mode = c->opt.tiles;
    a.mma = mma ? 1 : 0;
    a.btab = b.btab;
    // FP16 needs the lag products inside its range: int16 products reach 2^31
    const int f = c->steps[k0].fmt;
    const bool fp16 = c->opt.contract == DG_CONTRACT_FP16 || c->opt.contract == DG_CONTRACT_FP16X3;
    a.zscale = (mma && fp16 && f == DG_IQ_CI16) ? 1.0f / 65536.0f : 1.0f;
    a.wait_polls = g_tc_wait_polls.load(std::memory_order_relaxed);
}

static dg_status cdft_plan(dg_ctx *c, const CdftRun &r, const CdftBatch &a, size_t bi)
{
    CdftBufs &b = c->cd;
    const auto &bt = r.L->batches[bi];
    const bool mma = r.mma;
    const int kplan = r.refine ? DG_K_REFINE : DG_K_CDFT_PLAN;
    {
        Timed t(c, kplan);
        CK(c, launch_cdft_geo(a, c->stream));
        CK(c, cudaMemsetAsync(b.g2b, 0xff, sizeof(int4) * (size_t)bt.groups, c->stream));
        CK(c, launch_cdft_plan(a, (int)bt.nbt, c->stream));
        CK(c, launch_cdft_tiles(a, c->stream));
        t.done(mma ? 6 : 7);
    }
    return DG_OK;
}

// The batch's contraction; btab_only: only the tensor cores' DFT operand
// tables (the contraction itself then runs in a launch shared by several
// contexts).
static dg_status cdft_contract(dg_ctx *c, const CdftRun &r, const CdftBatch &a, size_t bi, bool btab_only)
{
    CdftBufs &b = c->cd;
    const auto &bt = r.L->batches[bi];
    const int k0 = bt.k0, S = bt.S, M = r.Ms[bi];
    const bool mma = r.mma, refine = r.refine;
    const CdftLayout &L = *r.L;
    const int f = c->steps[k0].fmt;
    if (btab_only) {
        Timed t(c, refine ? DG_K_REFINE : DG_K_CDFT_CONTRACT);
        CK(c, launch_cdft_btab(a, c->opt.contract, b.btab, c->stream));
        t.done(1);
        return DG_OK;
    }
    {
        Timed t(c, refine ? DG_K_REFINE : DG_K_CDFT_CONTRACT);
        if (mma) {
            // persistent: one CTA per SM, or fewer when the batch can
            // have fewer tiles (the bound: lag tiles of every lag slot)
            int64_t tiles_cap = 0;
            for (int s = 0; s < S; ++s) {
                const int slots = lag_slots(c->eph_host[k0 + s], c->fs, L.diam);
                const int64_t B = (c->steps[k0 + s].n + M - 1) / M;
                tiles_cap += B * ((slots + 127) / 128);
            }
            const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles_cap, c->sm_count));
            // Hankel tiles (chunk <= 1024, on request) run in their own
            // persistent kernel
            const bool hk = M <= kLagTileMaxChunk && c->opt.tiles == DG_TILES_HANKEL;
            int n = 0;
            if (c->opt.tiles != DG_TILES_HANKEL || M > kLagTileMaxChunk) {
                CK(c, launch_cdft_btab(a, c->opt.contract, b.btab, c->stream));
                CK(c, launch_cdft_contract_mma(a, grid, f, c->opt.contract, c->stream));
                n += 2;
            }
            if (hk) {
                int64_t hk_cap = 0;
                for (int s = 0; s < S; ++s) {
                    const int slots = lag_slots(c->eph_host[k0 + s], c->fs, L.diam);
                    const int64_t B = (c->steps[k0 + s].n + M - 1) / M;
                    hk_cap += B * ((slots + kHkLags - 1) / kHkLags);
                }
                const int hgrid = (int)std::max<int64_t>(1, std::min<int64_t>(hk_cap, c->sm_count));
                CK(c, launch_cdft_contract_hankel(a, hgrid, f, c->opt.contract, c->stream));
                ++n;
            }
            t.done(n);
        } else {
            CK(c, launch_cdft_contract_fp32(a, (int)bt.nbt, f, c->stream));
            t.done(1);
        }
    }
    return DG_OK;
}

static dg_status cdft_combine(dg_ctx *c, const CdftRun &r, const CdftBatch &a, size_t bi)
{
    const auto &bt = r.L->batches[bi];
    const bool refine = r.refine;
    float *surf_f = reinterpret_cast<float *>(r.surf);
    {
        Timed t(c, refine ? DG_K_REFINE : DG_K_CDFT_COMBINE);
        CK(c, launch_cdft_superchunk(a, (int)bt.nbt, c->stream));
        CK(c, launch_cdft_combine(a, surf_f, c->stream));
        t.done(2);
    }
    return DG_OK;
}

static dg_status cdft_finish(dg_ctx *c, const CdftRun &r)
{
    const bool refine = r.refine;
    {
        Timed t(c, refine ? DG_K_REFINE : DG_K_ACCUM);
        CK(c, launch_accumulate(r.surf, c->K, r.G, DG_PREC_FP32, r.out, c->stream));
        t.done(1);
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    return DG_OK;
}

// ---------------------------------------------------------------------------
// Delay-Doppler maps (dg_map.cu): the plan of a context's main grid, made on
// the host from the grid, the ephemerides and the capture lengths only, and
// the surface.
// ---------------------------------------------------------------------------

// Doppler nodes of a block of Mb samples over a band of half width w: the
// Chebyshev interpolant of e^{j 2 pi nu m}, |nu| <= w, |m| <= Mb / 2, is off by
// at most 4 (theta / 2)^P / P!, theta = pi w Mb (the tail of its Bessel
// coefficients). 0 if more than kMapMaxNodes would be needed.
static int map_nodes(double halfw, int Mb)
{
    const double x = 0.5 * kPi * halfw * Mb;
    double term = 4.0;
    for (int P = 1; P <= kMapMaxNodes; ++P) {
        term *= x / P;
        if (P >= 2 && P > x && term <= 2e-7) return P;
    }
    return 0;
}

// Polynomial geometry (k_map_poly): the sample nodes of a tile of `rows`
// rows, and the least-squares matrix [kPolyTerms][kPolyPts] from their values
// to the coefficients of x^e y^b, e + b <= 5, of the offsets normalised to
// [-1, 1] (x rows, y columns).
static PolyShape poly_shape(int rows)
{
    static const int at64[6] = {1, 9, 23, 40, 54, 62}, at32[6] = {0, 4, 11, 20, 27, 31};
    PolyShape s{};
    s.rows = rows;
    int n = 0;
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) {
            if ((i == 0 || i == 5) && (j == 0 || j == 5)) continue;
            s.pr[n] = (rows == 64 ? at64 : at32)[i];
            s.pc[n++] = at32[j];
        }
    return s;
}

static std::vector<float> poly_fit(const PolyShape &s)
{
    double A[kPolyPts][kPolyTerms], N[kPolyTerms][kPolyTerms + kPolyPts];
    for (int i = 0; i < kPolyPts; ++i) {
        const double x = (s.pr[i] - 0.5 * (s.rows - 1)) / (0.5 * (s.rows - 1));
        const double y = (s.pc[i] - 0.5 * (kPolyCols - 1)) / (0.5 * (kPolyCols - 1));
        int t = 0;
        for (int e = 0; e < 6; ++e)
            for (int b = 0; b + e < 6; ++b) A[i][t++] = std::pow(x, e) * std::pow(y, b);
    }
    for (int t = 0; t < kPolyTerms; ++t) {
        for (int u = 0; u < kPolyTerms; ++u) {
            N[t][u] = 0.0;
            for (int i = 0; i < kPolyPts; ++i) N[t][u] += A[i][t] * A[i][u];
        }
        for (int i = 0; i < kPolyPts; ++i) N[t][kPolyTerms + i] = A[i][t];
    }
    // normal equations N X = A^T by Gauss-Jordan elimination with pivoting
    for (int t = 0; t < kPolyTerms; ++t) {
        int piv = t;
        for (int u = t + 1; u < kPolyTerms; ++u)
            if (std::fabs(N[u][t]) > std::fabs(N[piv][t])) piv = u;
        for (int k = 0; k < kPolyTerms + kPolyPts; ++k) std::swap(N[t][k], N[piv][k]);
        const double d = 1.0 / N[t][t];
        for (int k = 0; k < kPolyTerms + kPolyPts; ++k) N[t][k] *= d;
        for (int u = 0; u < kPolyTerms; ++u) {
            if (u == t) continue;
            const double f = N[u][t];
            for (int k = 0; k < kPolyTerms + kPolyPts; ++k) N[u][k] -= f * N[t][k];
        }
    }
    std::vector<float> fit((size_t)kPolyTerms * kPolyPts);
    for (int t = 0; t < kPolyTerms; ++t)
        for (int i = 0; i < kPolyPts; ++i) fit[(size_t)t * kPolyPts + i] = (float)N[t][kPolyTerms + i];
    return fit;
}

// Tile rows of the polynomial geometry, or 0 (geometry per node): the grid
// must fill the chip with tiles, its slopes stay under 8 samples per node
// (exact linear part), and the bound on the first dropped terms, with a factor
// 4 for the fit and 2^5 for the Chebyshev-like samples, under 2e-6 samples and
// bins (1e-7 samples with the fractional delay, which uses D's fraction).
static int poly_rows(const dg_ctx *c, const std::vector<MapSnap> &snap)
{
    const bool frac = c->opt.delay != DG_DELAY_INTEGER;
    const int64_t tj = (c->gd.nlon + kPolyCols - 1) / kPolyCols;
    for (int rows : {64, 32}) {
        if (c->gd.nrows < rows || c->gd.nlon < kPolyCols) continue;
        if (tj * ((c->gd.nrows + rows - 1) / rows) < (int64_t)c->sm_count * (rows == 64 ? 8 : 2)) continue;
        bool ok = true;
        for (int k = 0; k < c->K && ok; ++k) {
            const GridRange &R = c->cd.main_range[k];
            const double B = R.sep * c->fs / kC;
            const double h = std::hypot(0.5 * rows * R.row_m, 0.5 * kPolyCols * R.col_m) / R.rho;
            const double h6 = h * h * h * h * h * h;
            const double u = R.vel * R.sep / (R.rho * c->lambda * c->fs * snap[k].delta);
            ok = B / R.rho * std::max(R.row_m, R.col_m) < 8.0 && B * 6.0 * h6 / 8.0 < (frac ? 1e-7 : 2e-6) &&
                 u * 36.0 * h6 / 8.0 < 2e-6;
        }
        if (ok) return rows;
    }
    return 0;
}

// The tables of `snap` (table s of capture s % K over lag and FDOA bounds
// range[s]) share one shape. Sets L0, NL and the bins of every table and
// Q, P, n = 2^logn, the lag tile LT and the block Mb = n - LT of m: those that
// take the fewest SM cycles by a model of the kernels (FFT butterflies at
// 0.35 of the FP32 rate, expansion at 0.5, a floor for the chain of one
// CTA). False where the captures or the ranges do not suit the maps.
static bool map_shape(const dg_ctx *c, const std::vector<GridRange> &range, std::vector<MapSnap> &snap, MapPlan &m)
{
    const bool frac = c->opt.delay != DG_DELAY_INTEGER;
    snap.assign(range.size(), MapSnap{});
    int nmax = 1, nlmax = 1;
    double Qd = 8.0;
    for (int k = 0; k < c->K; ++k) {
        if (c->steps[k].n > (1 << 24)) return false;
        nmax = std::max(nmax, (int)c->steps[k].n);
        m.c64 |= c->steps[k].fmt == DG_IQ_C64;
    }
    for (size_t s = 0; s < range.size(); ++s) {
        const GridRange &R = range[s];
        // 0.01 samples absorb the rounding of D; Lagrange4 reaches L - 1 .. L + 2
        if (!(std::fabs(R.d_lo) < 4e6 && std::fabs(R.d_hi) < 4e6)) return false;
        const int lo = (int)std::floor(R.d_lo - 0.51) - (frac ? 1 : 0), hi = (int)std::ceil(R.d_hi + 0.51) + (frac ? 2 : 0);
        snap[s].L0 = lo;
        snap[s].NL = hi - lo + 1;
        nlmax = std::max(nlmax, snap[s].NL);
        const double w = (R.nu_hi - R.nu_lo) * (1.0 + 1e-5) + 1e-13;
        if (!(w < 0.046)) return false;  // wider than the 64 bins of the contraction's shortest chunk take: refused there
        Qd = std::max(Qd, 6.0 + std::ceil(w * (double)c->steps[s % c->K].n / kMapNDelta));
    }
    if (Qd > 8192.0 || nlmax > 65536) return false;
    m.Q = (int)Qd;
    double halfw = 0.0;
    for (size_t q = 0; q < range.size(); ++q) {
        MapSnap &s = snap[q];
        const GridRange &R = range[q];
        s.delta = ((R.nu_hi - R.nu_lo) * (1.0 + 1e-5) + 1e-13) / (m.Q - 6);
        s.nu0 = 0.5 * (R.nu_lo + R.nu_hi) - 0.5 * (m.Q - 1) * s.delta;
        s.nuc = 0.5 * (R.nu_lo + R.nu_hi);
        s.halfw = 0.5 * (m.Q - 1) * s.delta;
        s.nu0_hi = (float)s.nu0;
        s.nu0_lo = (float)(s.nu0 - (double)s.nu0_hi);
        s.inv_delta = (float)(1.0 / s.delta);
        s.inv_delta_lo = (float)(1.0 / s.delta - (double)s.inv_delta);
        halfw = std::max(halfw, s.halfw);
    }
    std::map<int64_t, int> lengths;  // tables of each capture length
    for (int k = 0; k < c->K; ++k) lengths[c->steps[k].n] += (int)(range.size() / (size_t)c->K);
    double best = 1e300;
    for (int logn = 10; logn <= 14; ++logn) {
        const int n = 1 << logn;
        for (int nt = 1; nt <= 64; ++nt) {
            int LT = (nlmax + nt - 1) / nt;
            LT = (LT + 31) / 32 * 32;
            const int Mb = (n - LT) & ~1;
            if (Mb < n / 8) continue;
            const int P = map_nodes(halfw, Mb);
            if (P == 0) continue;
            double blocks = 0.0;
            for (const auto &l : lengths) blocks += std::ceil((double)l.first / Mb) * l.second;
            const double cmax = std::ceil((double)nmax / Mb), ffts = blocks * nt * (1 + 2 * P);
            const double exps = blocks * nlmax * m.Q * (2 * P + 4);
            const double t_fft = ffts * n * logn * 5.0 / (128 * 0.35) / c->sm_count;
            const double cost = std::max(t_fft, 3.0 * (4000.0 + 1.6 * n)) + exps / (128 * 0.5) / c->sm_count +
                                cmax * P * 40.0;
            if (cost < best) {
                best = cost;
                m.logn = logn;
                m.Mb = Mb;
                m.LT = LT;
                m.P = P;
            }
            if (nt * 32 >= nlmax) break;
        }
    }
    if (best == 1e300) return false;
    m.ntile = (nlmax + m.LT - 1) / m.LT;
    m.NLpad = (nlmax + 31) / 32 * 32;
    m.Cmax = (nmax + m.Mb - 1) / m.Mb;
    for (int p = 0; p < m.P; ++p) m.xnode[p] = std::cos(kPi * (p + 0.5) / m.P);
    return true;
}

// Device memory of one table (bytes) and of S of them at a time; the captures'
// tables `snap` and the node polynomials (never inside a captured graph: a
// graph is captured after one uncaptured call of the same shape).
static double map_bytes(const MapPlan &m)
{
    return 8.0 * ((double)m.ntile * m.Cmax * ((size_t)1 << m.logn) + (double)m.Cmax * m.P * m.NLpad +
                  (double)m.Q * m.NLpad + (double)m.Cmax * m.Q);
}
static dg_status map_buffers(dg_ctx *c, const MapPlan &m, size_t S, const std::vector<MapSnap> &snap)
{
    MapBufs &d = c->mb;
    const size_t n = (size_t)1 << m.logn;
    dg_status st;
    if ((st = ensure(c, (void **)&d.snap, &d.snap_cap, sizeof(MapSnap) * snap.size())) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.tw, &d.tw_cap, sizeof(float2) * n, &d.tw_logn)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.T, &d.T_cap, sizeof(float) * (size_t)m.P * m.Q, &d.T_P)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.F2, &d.F2_cap, sizeof(float2) * S * m.ntile * m.Cmax * n)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.U, &d.U_cap, sizeof(float2) * S * m.Cmax * m.P * m.NLpad)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.X, &d.X_cap, sizeof(float2) * S * m.Q * m.NLpad)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.phase, &d.phase_cap, sizeof(float2) * S * m.Cmax * m.Q)) != DG_OK) return st;
    if (m.c64 && (st = ensure(c, (void **)&d.bad, &d.bad_cap, sizeof(int) * 4 * (size_t)c->K)) != DG_OK) return st;
    if ((st = ensure_ephf(c)) != DG_OK) return st;
    // pageable sources: staged before the calls return
    CK(c, cudaMemcpyAsync(d.snap, snap.data(), sizeof(MapSnap) * snap.size(), cudaMemcpyHostToDevice, c->stream));
    if (d.tw_logn != m.logn) {
        d.tw_logn = 0;
        CK(c, launch_map_twiddles(d.tw, m.logn, c->stream));
        ++c->launches;
        d.tw_logn = m.logn;
    }
    if (d.T_P != m.P || d.T_Q != m.Q) {
        std::vector<float> T((size_t)m.P * m.Q);
        for (int p = 0; p < m.P; ++p)
            for (int q = 0; q < m.Q; ++q) {
                const double x = -1.0 + 2.0 * q / (m.Q - 1);
                double t = 1.0;
                for (int r = 0; r < m.P; ++r)
                    if (r != p) t *= (x - m.xnode[r]) / (m.xnode[p] - m.xnode[r]);
                T[(size_t)p * m.Q + q] = (float)t;
            }
        d.T_P = 0;
        CK(c, cudaMemcpyAsync(d.T, T.data(), sizeof(float) * T.size(), cudaMemcpyHostToDevice, c->stream));
        d.T_P = m.P;
        d.T_Q = m.Q;
    }
    return DG_OK;
}

// The chunk the contraction would take for the context's grid (what
// dg_cdft_chunks reports whichever way the surface is computed), and whether
// its per-lag DFT buffer would stay within the limit of cdft_setup.
static bool map_chunks(dg_ctx *c, int *lo, int *hi)
{
    CdftBufs &b = c->cd;
    if (b.main_span.size() != (size_t)c->K || b.main_lags.size() != (size_t)c->K ||
        b.main_range.size() != (size_t)c->K)
        fdoa_spans(c, c->gd, b.main_span, &b.main_lags, &b.main_range);
    CdftLayout L;
    std::vector<int> bb, gb;
    if (cdft_batches(c, c->G, grid_diameter(c->gd), L, bb, gb) != DG_OK) return false;
    const bool tc = c->opt.contract != DG_CONTRACT_FP32;
    *lo = INT_MAX;
    *hi = 0;
    int64_t B = 1;
    for (const auto &t : L.batches) {
        const int M = auto_chunk(c, b.main_span, b.main_lags, t.k0, t.S, tc);
        *lo = std::min(*lo, M);
        *hi = std::max(*hi, M);
        for (int s = 0; s < t.S; ++s) B = std::max<int64_t>(B, (c->steps[t.k0 + s].n + M - 1) / M);
    }
    return (double)L.nbt_max * (double)B * 512.0 <= (double)((size_t)64 << 30);
}

static dg_status make_map_plan(dg_ctx *c)
{
    MapPlan &m = c->mp;
    CdftBufs &b = c->cd;
    if (!map_chunks(c, &m.chunk_min, &m.chunk_max)) return DG_OK;
    std::vector<MapSnap> snap;
    if (!map_shape(c, b.main_range, snap, m)) return DG_OK;
    for (int k = 0; k < c->K; ++k) m.rows += (int64_t)snap[k].NL * ((c->steps[k].n + m.Mb - 1) / m.Mb);
    const int pr = poly_rows(c, snap);
    if (pr) m.poly = poly_shape(pr);
    const double ptiles = pr ? std::ceil((double)c->gd.nrows / pr) * std::ceil((double)c->gd.nlon / kPolyCols) : 0.0;
    const double per = map_bytes(m) + 4.0 * kPolyStride * ptiles;
    const double budget = (double)(c->opt.scratch_mib ? c->opt.scratch_mib : 12288) * 1048576.0;
    m.S = (int)std::max(1.0, std::min((double)c->K, std::floor(budget / per)));
    dg_status st;
    if (pr) {
        MapBufs &d = c->mb;
        const size_t fb = sizeof(float) * kPolyTerms * kPolyPts;
        if ((st = ensure(c, (void **)&d.fit, &d.fit_cap, fb, &d.fit_rows)) != DG_OK) return st;
        if ((st = ensure(c, (void **)&d.coef, &d.coef_cap, sizeof(float) * kPolyStride * (size_t)ptiles * m.S)) != DG_OK)
            return st;
        if (d.fit_rows != pr) {
            const std::vector<float> fit = poly_fit(m.poly);
            d.fit_rows = 0;
            CK(c, cudaMemcpyAsync(d.fit, fit.data(), fb, cudaMemcpyHostToDevice, c->stream));
            d.fit_rows = pr;
        }
    }
    if ((st = map_buffers(c, m, (size_t)m.S, snap)) != DG_OK) return st;
    m.ok = true;
    return DG_OK;
}
static dg_status map_plan(dg_ctx *c)
{
    if (c->mp.gen == c->steps_gen) return DG_OK;
    c->mp = MapPlan{};
    const dg_status st = make_map_plan(c);
    // tables or not, the outcome holds until the shapes change; an error is tried again
    if (st == DG_OK) c->mp.gen = c->steps_gen;
    return st;
}

// The arguments every table shares: captures and ephemerides from snapshot k0
// on, the grid, the geometry's constants.
static void map_common(dg_ctx *c, int k0, const double *xyz, const GridDev &gd, int64_t G, MapArgs &a)
{
    auto split = [](double v, float &h, float &l) {
        h = (float)v;
        l = (float)(v - (double)h);
    };
    a.sd = c->steps_d + k0;
    a.xyz = xyz;
    a.eph = c->eph + 12 * (size_t)k0;
    a.ephf = c->cd.ephf + 24 * (size_t)k0;
    split(c->fs / kC, a.fsc_hi, a.fsc_lo);
    split(1.0 / (c->lambda * c->fs), a.ilf_hi, a.ilf_lo);
    a.fs = c->fs;
    a.lambda = c->lambda;
    a.G = G;
    a.nrows = gd.nrows;
    a.nlon = gd.nlon;
    a.delay = c->opt.delay;
    a.acc = c->opt.acc;
    a.err = c->err_d;
    a.nreg = 1;
}

// The shape and the scratch of a plan's tables.
static void map_tables_args(const MapPlan &m, const MapBufs &d, MapArgs &a)
{
    a.logn = m.logn;
    a.Mb = m.Mb;
    a.Cmax = m.Cmax;
    a.P = m.P;
    a.Q = m.Q;
    a.LT = m.LT;
    a.ntile = m.ntile;
    a.NLpad = m.NLpad;
    a.tw = d.tw;
    a.T = d.T;
    std::memcpy(a.xnode, m.xnode, sizeof a.xnode);
    a.F2 = d.F2;
    a.U = d.U;
    a.X = d.X;
    a.phase = d.phase;
    a.bad = m.c64 ? d.bad : nullptr;
}

static dg_status run_surface_map(dg_ctx *c, void *out)
{
    const MapPlan &m = c->mp;
    MapBufs &d = c->mb;
    dg_status st = push_steps(c);
    if (st != DG_OK) return st;
    c->cd_chunk_min = m.chunk_min;
    c->cd_chunk_max = m.chunk_max;
    c->last_map = true;
    for (int k0 = 0; k0 < c->K; k0 += m.S) {
        MapArgs a{};
        map_common(c, k0, c->xyz, c->gd, c->G, a);
        a.S = a.ksd = std::min(m.S, c->K - k0);
        a.snap = d.snap + k0;
        map_tables_args(m, d, a);
        a.first = k0 == 0;
        a.out = (float *)out;
        a.poly = m.poly;
        a.fit = d.fit;
        a.coef = d.coef;
        if (m.poly.rows) {
            Timed t(c, DG_K_CDFT_COMBINE);
            CK(c, launch_map_poly(a, c->stream));
            t.done(1);
        }
        {
            Timed t(c, DG_K_CDFT_CONTRACT);
            int n = 1;
            CK(c, launch_map_tables(a, c->stream, &n));
            CK(c, launch_map_expand(a, c->stream));
            t.done(n);
        }
        {
            Timed t(c, DG_K_CDFT_COMBINE);
            CK(c, launch_map_lookup(a, c->stream));
            t.done(1);
        }
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    return DG_OK;
}

// The least distance between the grid's nodes and the receivers of any
// snapshot, less half the receivers' separation (0: no bound), and the
// largest separation and relative motion. From 3 x 3 nodes where the grid is
// small against its range (half a cell off at most), else 17 x 17.
struct RefineBound {
    double rho = 1e300, sep = 0.0, vel = 0.0, dv = 0.0;
};
static RefineBound refine_bound(const dg_ctx *c, const GridDev &g)
{
    for (int side : {3, 17}) {
        RefineBound b;
        const int ni = std::min(side, g.nrows), nj = std::min(side, g.nlon);
        std::vector<double> p(3 * (size_t)ni * nj);
        for (int i = 0; i < ni; ++i)
            for (int j = 0; j < nj; ++j)
                host_node_ecef(g, g.row0 + (ni > 1 ? (double)i * (g.nrows - 1) / (ni - 1) : 0.0),
                               nj > 1 ? (double)j * (g.nlon - 1) / (nj - 1) : 0.0, &p[3 * ((size_t)i * nj + j)]);
        auto norm = [](double x, double y, double z) { return std::sqrt(x * x + y * y + z * z); };
        double hi = 0.0, hj = 0.0, rmin = 1e300;
        for (int i = 0; i < ni; ++i)
            for (int j = 0; j < nj; ++j) {
                const double *x = &p[3 * ((size_t)i * nj + j)];
                if (i + 1 < ni) hi = std::max(hi, norm(x[0] - x[3 * nj], x[1] - x[3 * nj + 1], x[2] - x[3 * nj + 2]));
                if (j + 1 < nj) hj = std::max(hj, norm(x[0] - x[3], x[1] - x[4], x[2] - x[5]));
                for (int k = 0; k < c->K; ++k) {
                    const dg_ephem &e = c->eph_host[k];
                    rmin = std::min(rmin, std::min(norm(e.p1[0] - x[0], e.p1[1] - x[1], e.p1[2] - x[2]),
                                                   norm(e.p2[0] - x[0], e.p2[1] - x[1], e.p2[2] - x[2])));
                }
            }
        for (int k = 0; k < c->K; ++k) {
            const dg_ephem &e = c->eph_host[k];
            b.sep = std::max(b.sep, norm(e.p2[0] - e.p1[0], e.p2[1] - e.p1[1], e.p2[2] - e.p1[2]));
            b.dv = std::max(b.dv, norm(e.v2[0] - e.v1[0], e.v2[1] - e.v1[1], e.v2[2] - e.v1[2]));
            b.vel = std::max(b.vel, std::max(norm(e.v1[0], e.v1[1], e.v1[2]), norm(e.v2[0], e.v2[1], e.v2[2])));
        }
        const double h = 0.55 * std::hypot(hi, hj);
        b.rho = rmin - h - 0.5 * b.sep;
        if (b.rho > 0.75 * rmin || side == 17) return b;
    }
    return RefineBound{};
}

// A refinement surface from a table of few lags (k_map_few), planned from the
// grid's shape and bounds that hold anywhere on the main grids (its centre, a node
// of one of them, is known on the device only). *done = false where the shape does
// not suit it.
static dg_status refine_map(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *out, bool *done,
                            const GridDev *mains, int nmains)
{
    *done = false;
    if (!(gd.nlat & 1) || gd.nlat != gd.nlon || gd.nrows != gd.nlat) return DG_OK;  // the centre is a node
    int nmax = 1;
    bool c64 = false;
    for (int k = 0; k < c->K; ++k) {
        if (c->steps[k].n > (1 << 24) || !c->steps[k].loaded) return DG_OK;
        nmax = std::max(nmax, (int)c->steps[k].n);
        c64 |= c->steps[k].fmt == DG_IQ_C64;
    }
    // the farthest node: half a diagonal of the lattice in metres, with 2 % for
    // the parallels' change of radius over up to 20 km at 80 degrees
    RefineBound rb;
    for (int i = 0; i < nmains; ++i) {
        if (std::fabs(mains[i].lat0_rad) + 0.5 * mains[i].nlat * mains[i].dlat_m / 6.33e6 > 1.39 || lon_extent(mains[i]) > 3.0)
            return DG_OK;
        const RefineBound q = refine_bound(c, mains[i]);
        const double rho = std::min(rb.rho, q.rho);
        rb = q;
        rb.rho = rho;
    }
    const double half = (gd.nlat - 1) / 2, r = 1.02 * half * std::hypot(gd.dlat_m, gd.dlon_m);
    const double rho = rb.rho - r;
    if (!(rho > 0.0) || r > 2e4) return DG_OK;
    const double md = rb.sep / rho * c->fs / kC * r;
    const double mn = (rb.dv / rho + 3.0 * rb.vel * rb.sep / (rho * rho)) / (c->lambda * c->fs) * r;
    const bool frac = c->opt.delay != DG_DELAY_INTEGER;
    const double nl = std::ceil(2.0 * md + 1.02) + 2.0 + (frac ? 3.0 : 0.0);
    const double w = 2.0 * mn * (1.0 + 1e-5) + 1e-13;
    // the most bins the tables hold: the six that pad the stencils then widen the
    // band least (at 8 bins it would be 3.5 times the FDOAs' own)
    if (nl > kFewMaxLags || 6.0 + std::ceil(w * nmax / kMapNDelta) > kFewMaxBins) return DG_OK;
    MapArgs a{};
    MapFew f{};
    a.Q = kFewMaxBins;
    a.LT = (int)nl;
    f.delta = w / (a.Q - 6);
    f.halfw = 0.5 * (a.Q - 1) * f.delta;
    f.md = md;
    f.centre = (G - 1) / 2;
    // terms of the Chebyshev series over the longest capture (the tail is at
    // most 2 |J_P(theta)|: map_nodes' bound, for capture = block)
    const int need = map_nodes(f.halfw, nmax);
    if (need == 0 || need > kFewMaxNodes) return DG_OK;
    a.P = need <= 4 ? 4 : need <= 6 ? 6 : 8;
    a.NLpad = 32;
    a.S = a.ksd = c->K;
    f.tscale = 2.0f / (float)(nmax + 1);
    // CTAs per snapshot: what fits on the chip over all snapshots (by the kernel's
    // registers), a block of samples each at least
    const int per_sm = a.P == 4 ? 4 : a.P == 6 ? 3 : 2;
    a.Cmax = std::max(1, std::min((nmax + kFewBlock - 1) / kFewBlock, per_sm * c->sm_count / c->K));
    const size_t u = sizeof(float) * map_few_partials(a.P, a.LT) * (size_t)a.Cmax * c->K;
    if (u > ((size_t)1 << 32) || (c->opt.scratch_mib && (double)u > c->opt.scratch_mib * 1048576.0)) return DG_OK;
    dg_status st = push_steps(c);
    if (st != DG_OK) return st;
    MapBufs &d = c->mr;
    if ((st = ensure(c, (void **)&d.snap, &d.snap_cap, sizeof(MapSnap) * (size_t)c->K)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.U, &d.U_cap, u)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&d.X, &d.X_cap, sizeof(float2) * (size_t)c->K * a.Q * a.NLpad)) != DG_OK) return st;
    if (c64 && (st = ensure(c, (void **)&d.bad, &d.bad_cap, sizeof(int) * 4 * (size_t)c->K)) != DG_OK) return st;
    if ((st = ensure_ephf(c)) != DG_OK) return st;
    // e^{j theta_q t} = sum_m j^m T[m][q] T_m(t), theta_q the phase of bin q at
    // t = 1: the series' real coefficients by a 32-point cosine sum, folded (the
    // points lie symmetrically around 0, and so do the bins). 272 sines on the
    // host; each coefficient's own sum took 12 thousand, 90 us.
    double px[16], tm[kFewMaxNodes][16];  // points cos((i + 1/2) pi / 32), T_m there
    for (int i = 0; i < 16; ++i) {
        px[i] = std::cos(kPi * (i + 0.5) / 32.0);
        for (int m = 0; m < a.P; ++m)
            tm[m][i] = m == 0 ? 1.0 : m == 1 ? px[i] : 2.0 * px[i] * tm[m - 1][i] - tm[m - 2][i];
    }
    for (int q = 0; q < a.Q / 2; ++q) {
        const double theta = 2.0 * kPi * (q * f.delta - f.halfw) / f.tscale;
        double cs[16], sn[16];
        for (int i = 0; i < 16; ++i) {
            cs[i] = std::cos(theta * px[i]);
            sn[i] = std::sin(theta * px[i]);
        }
        for (int m = 0; m < a.P; ++m) {
            double x = 0.0;
            for (int i = 0; i < 16; ++i) x += (m & 1 ? sn[i] : cs[i]) * tm[m][i];
            x *= (m ? 4.0 : 2.0) / 32.0 * (m % 4 < 2 ? 1.0 : -1.0);
            f.T[m * a.Q + q] = (float)x;
            f.T[m * a.Q + a.Q - 1 - q] = (float)(m & 1 ? -x : x);
        }
    }
    map_common(c, 0, xyz, gd, G, a);
    f.snap = d.snap;
    a.snap = d.snap;
    a.first = 1;
    a.U = d.U;
    a.X = d.X;
    a.bad = c64 ? d.bad : nullptr;
    a.out = (float *)out;
    {
        Timed t(c, DG_K_REFINE);
        int n = 1;
        CK(c, launch_map_few(a, f, c->stream, &n));
        CK(c, launch_map_lookup(a, c->stream));
        t.done(n);
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    *done = true;
    return DG_OK;
}

// The per-snapshot surfaces [K][G] of a main surface (the maps need none).
static dg_status ensure_surf(dg_ctx *c)
{
    if (map_eligible(c)) {
        const dg_status st = map_plan(c);
        if (st != DG_OK || c->mp.ok) return st;
    }
    const size_t esz = c->opt.prec == DG_PREC_FP64 ? 8 : 4;
    return ensure(c, &c->surf, &c->surf_bytes, esz * (size_t)c->G * c->K);
}

dg_status run_surface_cdft(dg_ctx *c, const GridDev &gd, const double *xyz, int64_t G, void *surf, void *out,
                           bool refine)
{
    CdftRun r;
    if (!refine) c->last_map = false;
    r.gd = gd;
    r.xyz = xyz;
    r.G = G;
    r.surf = surf;
    r.out = out;
    r.refine = refine;
    dg_status st = cdft_setup(c, r);
    if (st != DG_OK) return st;
    for (size_t bi = 0; bi < r.L->batches.size(); ++bi) {
        CdftBatch a{};
        cdft_args(c, r, bi, a);
        if ((st = cdft_plan(c, r, a, bi)) != DG_OK) return st;
        if ((st = cdft_contract(c, r, a, bi, false)) != DG_OK) return st;
        if ((st = cdft_combine(c, r, a, bi)) != DG_OK) return st;
    }
    return cdft_finish(c, r);
}

dg_status run_argmax(dg_ctx *c, const void *v, int64_t n, const GridDev &gd, ArgmaxResult *host)
{
    size_t need = argmax_tmp_bytes(n);
    dg_status st = ensure(c, &c->amax_tmp, &c->amax_tmp_bytes, need);
    if (st != DG_OK) return st;
    int nlaunch = 0;
    {
        Timed t(c, DG_K_ARGMAX);
        CK(c, launch_argmax(v, n, c->opt.prec, gd, c->gstep, c->amax_tmp, c->amax_res, &nlaunch, c->stream));
        t.done(nlaunch);
    }
    CK(c, cudaMemcpyAsync(c->amax_host, c->amax_res, sizeof(ArgmaxResult), cudaMemcpyDeviceToHost,
                          c->stream));
    CK(c, cudaStreamSynchronize(c->stream));
    *host = *c->amax_host;
    return DG_OK;
}

GridDev make_griddev(const dg_grid &g, int row0, int nrows)
{
    GridDev d;
    d.lat0_rad = g.lat0_deg * (kPi / 180.0);
    d.lon0_rad = g.lon0_deg * (kPi / 180.0);
    d.dlat_m = g.dlat_m;
    d.dlon_m = g.dlon_m;
    d.nlat = g.nlat;
    d.nlon = g.nlon;
    d.row0 = row0;
    d.nrows = nrows;
    return d;
}

dg_status validate_grid(dg_ctx *c, const dg_grid *g)
{
    if (!g) return fail(c, DG_EINVAL, "grid is NULL");
    if (!(std::isfinite(g->lat0_deg) && std::fabs(g->lat0_deg) < 89.0))
        return fail(c, DG_EINVAL, "lat0_deg must be finite and within +-89 deg");
    if (!std::isfinite(g->lon0_deg)) return fail(c, DG_EINVAL, "lon0_deg must be finite");
    if (!(g->dlat_m > 0 && g->dlon_m > 0 && std::isfinite(g->dlat_m) && std::isfinite(g->dlon_m)))
        return fail(c, DG_EINVAL, "grid spacing must be positive and finite");
    if (g->nlat < 1 || g->nlon < 1) return fail(c, DG_EINVAL, "nlat and nlon must be >= 1");
    if ((int64_t)g->nlat * g->nlon > (int64_t)1 << 31)
        return fail(c, DG_EUNSUPPORTED, "grid larger than 2^31 nodes");
    return DG_OK;
}

}  // namespace

extern "C" {

int32_t dg_abi_version(void) { return DG_ABI_VERSION; }

void dg_options_default(dg_options *o)
{
    if (!o) return;
    std::memset(o, 0, sizeof *o);
    o->delay = DG_DELAY_INTEGER;
    o->acc = DG_ACC_POWER;
    o->prec = DG_PREC_FP32;
    o->algo = DG_ALGO_DIRECT;
}

const char *dg_last_error(const dg_ctx *ctx) { return ctx ? ctx->err.c_str() : g_thread_error.c_str(); }

dg_status dg_create(const dg_grid *grid, const dg_ephem *eph, int32_t K, double fs_hz, double fc_hz,
                    const dg_options *opt, void *cuda_stream, dg_ctx **out)
{
    g_thread_error.clear();
    if (!out) return fail(nullptr, DG_EINVAL, "out is NULL");
    dg_status st = validate_grid(nullptr, grid);
    if (st != DG_OK) return st;
    if (!eph) return fail(nullptr, DG_EINVAL, "eph is NULL");
    if (K < 1 || K > 65535) return fail(nullptr, DG_EINVAL, "K must be in [1, 65535]");
    if (!(fs_hz > 0 && std::isfinite(fs_hz))) return fail(nullptr, DG_EINVAL, "fs_hz must be > 0");
    if (!(fc_hz > 0 && std::isfinite(fc_hz))) return fail(nullptr, DG_EINVAL, "fc_hz must be > 0");
    dg_options o;
    dg_options_default(&o);
    if (opt) o = *opt;
    if (o.delay != DG_DELAY_INTEGER && o.delay != DG_DELAY_LAGRANGE4)
        return fail(nullptr, DG_EINVAL, "unknown delay mode %d", o.delay);
    if (o.acc != DG_ACC_POWER && o.acc != DG_ACC_MAG) return fail(nullptr, DG_EINVAL, "unknown acc mode %d", o.acc);
    if (o.prec != DG_PREC_FP32 && o.prec != DG_PREC_FP64)
        return fail(nullptr, DG_EINVAL, "unknown precision %d", o.prec);
    if (o.algo != DG_ALGO_DIRECT && o.algo != DG_ALGO_CDFT) return fail(nullptr, DG_EINVAL, "unknown algorithm %d", o.algo);
    if (o.algo == DG_ALGO_CDFT) {
        if (o.prec != DG_PREC_FP32) return fail(nullptr, DG_EUNSUPPORTED, "CDFT writes FP32 surfaces only");
        if (o.chunk != 0 && (o.chunk < 64 || o.chunk > kCdftMaxChunk || o.chunk % 64 != 0))
            return fail(nullptr, DG_EINVAL, "chunk must be 0 or a multiple of 64 in [64, %d]", kCdftMaxChunk);
        if (o.bins != 0 && o.bins != 64) return fail(nullptr, DG_EUNSUPPORTED, "bins must be 0 or 64");
        if (o.contract < DG_CONTRACT_FP32 || o.contract > DG_CONTRACT_FP16X3)
            return fail(nullptr, DG_EINVAL, "unknown contraction arithmetic %d", o.contract);
        if (o.tiles < DG_TILES_AUTO || o.tiles > DG_TILES_HANKEL)
            return fail(nullptr, DG_EINVAL, "unknown tile shape %d", o.tiles);
        if (o.tiles == DG_TILES_HANKEL && o.chunk > kLagTileMaxChunk)
            return fail(nullptr, DG_EINVAL, "Hankel tiles need chunk <= %d", kLagTileMaxChunk);
        if (o.tiles == DG_TILES_LAGS && o.chunk > kLagTileMaxChunk && o.chunk % kLagTileMaxChunk != 0)
            return fail(nullptr, DG_EINVAL, "lag tiles need chunk <= %d or a multiple of it", kLagTileMaxChunk);
        if (o.scratch_mib < 0) return fail(nullptr, DG_EINVAL, "scratch_mib must be >= 0");
    }
    if (!direct_rows_ok(o.prec, o.rows))
        return fail(nullptr, DG_EINVAL, "rows must be 0, 4, 8 or 16 (FP32) or 0, 2 or 4 (FP64)");
    if (o.row0 < 0 || o.row0 >= grid->nlat) return fail(nullptr, DG_EINVAL, "row0 outside the grid");
    if (o.nrows < 0 || o.row0 + o.nrows > grid->nlat) return fail(nullptr, DG_EINVAL, "row shard outside the grid");
    for (int k = 0; k < K; ++k)
        if (!finite3(eph[k].p1) || !finite3(eph[k].v1) || !finite3(eph[k].p2) || !finite3(eph[k].v2))
            return fail(nullptr, DG_EINVAL, "ephemeris %d is not finite", k);

    dg_ctx *c = new (std::nothrow) dg_ctx();
    if (!c) return fail(nullptr, DG_ENOMEM, "host allocation failed");
    c->grid = *grid;
    c->opt = o;
    c->K = K;
    c->fs = fs_hz;
    c->fc = fc_hz;
    c->lambda = kC / fc_hz;
    c->stream = (cudaStream_t)cuda_stream;
    const int nrows = o.nrows ? o.nrows : grid->nlat - o.row0;
    c->gd = make_griddev(*grid, o.row0, nrows);
    c->G = (int64_t)nrows * grid->nlon;
    c->eph_host.assign(eph, eph + K);
    c->steps.resize(K);
    c->steps_h.resize(K);

    auto bail = [&](dg_status s) {
        g_thread_error = c->err;
        dg_destroy(c);
        return s;
    };
#define CKC(call)                                                                              \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return bail(fail(c, e_ == cudaErrorMemoryAllocation ? DG_ENOMEM : DG_ECUDA, "%s: %s", \
                             #call, cudaGetErrorString(e_)));                                  \
    } while (0)
    CKC(cudaGetDevice(&c->device));
    CKC(cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device));
    CKC(device_alloc(c, &c->xyz, sizeof(double) * 3 * (size_t)c->G));
    c->xyz_cap = c->G;
    CKC(device_alloc(c, &c->gstep, 2 * sizeof(GridStep)));
    CKC(device_alloc(c, &c->eph, sizeof(double) * 12 * (size_t)K));
    CKC(device_alloc(c, &c->steps_d, sizeof(StepDesc) * (size_t)K));
    CKC(device_alloc(c, &c->amax_res, sizeof(ArgmaxResult)));
    CKC(device_alloc(c, &c->err_d, sizeof(unsigned)));
    CKC(pinned_alloc(&c->amax_host, sizeof(ArgmaxResult)));
    CKC(pinned_alloc(&c->err_h, sizeof(unsigned)));
    *c->err_h = 0;
    CKC(cudaMemsetAsync(c->err_d, 0, sizeof(unsigned), c->stream));
    CKC(cudaMemcpyAsync(c->eph, c->eph_host.data(), sizeof(dg_ephem) * (size_t)K, cudaMemcpyHostToDevice,
                        c->stream));
    {
        Timed t(c, DG_K_GRID);
        CKC(launch_grid_ecef(c->gd, c->xyz, c->stream, nullptr, nullptr, 1, c->gstep));
        t.done(1);
    }
    CKC(cudaStreamSynchronize(c->stream));  // eph_host may not move before the copy ran
#undef CKC
    *out = c;
    return DG_OK;
}

// The host's bounds of the current grid (fdoa_spans: 0.7 ms for a 65 x 65
// lattice and 20 snapshots) go to a list of the last few grids, by their values,
// and those of the next one come back from it: a search that alternates between a
// footprint and its regions computes each once.
static bool same_grid(const dg_grid &a, const dg_grid &b)
{
    return a.lat0_deg == b.lat0_deg && a.lon0_deg == b.lon0_deg && a.dlat_m == b.dlat_m && a.dlon_m == b.dlon_m &&
           a.nlat == b.nlat && a.nlon == b.nlon;
}
static void grid_bounds_switch(dg_ctx *c, const dg_grid &next)
{
    CdftBufs &b = c->cd;
    if (!b.main_span.empty()) {
        if (c->past.size() >= 4) c->past.erase(c->past.begin());
        c->past.push_back({c->grid, std::move(b.main_span), std::move(b.main_lags), std::move(b.main_range)});
    }
    b.main_span.clear();
    b.main_lags.clear();
    b.main_range.clear();
    for (size_t i = 0; i < c->past.size(); ++i) {
        if (!same_grid(c->past[i].grid, next)) continue;
        b.main_span = std::move(c->past[i].span);
        b.main_lags = std::move(c->past[i].lags);
        b.main_range = std::move(c->past[i].range);
        c->past.erase(c->past.begin() + (long)i);
        break;
    }
}

// xyz, step: the grid's nodes and angular steps where they are on the device.
static dg_status set_grid(dg_ctx *c, const dg_grid *grid, const double *xyz, const GridStep *step)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    dg_status st = validate_grid(c, grid);
    if (st != DG_OK) return st;
    if (c->gd.row0 != 0 || c->gd.nrows != c->grid.nlat)
        return fail(c, DG_EUNSUPPORTED, "dg_set_grid needs a context over the whole grid (no row shard)");
    const int64_t G = (int64_t)grid->nlat * grid->nlon;
    if (G > c->xyz_cap) {
        void *old = c->xyz;  // no nodes (need_nodes) until the new buffer is there
        c->xyz = nullptr;
        c->xyz_cap = 0;
        ++c->steps_gen;
        if ((st = release(c, old)) != DG_OK) return st;
        CK(c, device_alloc(c, &c->xyz, sizeof(double) * 3 * (size_t)G));
        c->xyz_cap = G;
    }
    const bool same = same_grid(c->grid, *grid);
    if (!same) grid_bounds_switch(c, *grid);
    c->grid = *grid;
    c->opt.row0 = 0;
    c->opt.nrows = 0;
    c->gd = make_griddev(*grid, 0, grid->nlat);
    c->G = G;
    ++c->steps_gen;           // graphs and batches recorded on the old grid are stale
    if (xyz) {
        CK(c, cudaMemcpyAsync(c->xyz, xyz, sizeof(double) * 3 * (size_t)G, cudaMemcpyDeviceToDevice, c->stream));
        CK(c, cudaMemcpyAsync(c->gstep, step, sizeof(GridStep), cudaMemcpyDeviceToDevice, c->stream));
        return DG_OK;
    }
    {
        Timed t(c, DG_K_GRID);
        CK(c, launch_grid_ecef(c->gd, c->xyz, c->stream, nullptr, nullptr, 1, c->gstep));
        t.done(1);
    }
    return DG_OK;
}

dg_status dg_set_grid(dg_ctx *c, const dg_grid *grid) { return set_grid(c, grid, nullptr, nullptr); }

dg_status dg_load_capture(dg_ctx *c, int32_t step, int32_t fmt, const void *y1, const void *y2,
                          int64_t n, int32_t is_device_ptr)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (step < 0 || step >= c->K) return fail(c, DG_EINVAL, "step %d outside [0, %d)", step, c->K);
    const size_t bps = iq_bytes(fmt);
    if (!bps) return fail(c, DG_EINVAL, "unknown IQ format %d", fmt);
    if (!y1 || !y2) return fail(c, DG_EINVAL, "y1 and y2 must not be NULL");
    if (n < 1) return fail(c, DG_EINVAL, "n_samples must be >= 1");
    if (n > ((int64_t)1 << 30)) return fail(c, DG_EUNSUPPORTED, "n_samples above 2^30");
    Step &s = c->steps[step];
    const size_t bytes = bps * (size_t)n;
    if (s.cap < bytes) {
        void *const old[2] = {s.y1, s.y2};
        s.y1 = s.y2 = nullptr;
        s.cap = 0;
        s.loaded = false;
        ++c->steps_gen;  // also where the allocation fails: captured steps read the old buffers
        for (void *p : old) {
            const dg_status st = release(c, p);
            if (st != DG_OK) return st;
        }
        CK(c, device_alloc(c, &s.y1, bytes));
        CK(c, device_alloc(c, &s.y2, bytes));
        s.cap = bytes;
    }
    const cudaMemcpyKind kind = is_device_ptr ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    CK(c, cudaMemcpyAsync(s.y1, y1, bytes, kind, c->stream));
    CK(c, cudaMemcpyAsync(s.y2, y2, bytes, kind, c->stream));
    if (s.fmt != fmt || s.n != n || !s.loaded) {
        c->steps_dirty = true;
        ++c->steps_gen;
    }
    s.fmt = fmt;
    s.n = n;
    s.loaded = true;
    return DG_OK;
}

dg_status dg_cost_surface(dg_ctx *c, void *out)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!out) return fail(c, DG_EINVAL, "out is NULL");
    for (int k = 0; k < c->K; ++k)
        if (!c->steps[k].loaded) return fail(c, DG_ESTATE, "snapshot %d has not been loaded", k);
    dg_status st = ensure_surf(c);
    if (st != DG_OK) return st;
    return run_surface(c, c->gd, c->xyz, c->G, c->surf, out, false);
}

dg_status dg_sync(dg_ctx *c)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    CK(c, cudaStreamSynchronize(c->stream));
    return check_latched(c);
}

// Buffers of a refinement grid of G nodes.
static dg_status ensure_local(dg_ctx *c, int64_t G)
{
    const size_t esz = c->opt.prec == DG_PREC_FP64 ? 8 : 4;
    if (c->loc.g_cap < (size_t)G) {
        dg_status st;
        if ((st = release(c, c->loc.xyz)) != DG_OK || (st = release(c, c->loc.surf)) != DG_OK ||
            (st = release(c, c->loc.cost)) != DG_OK)
            return st;
        c->loc = LocalGrid{};
        CK(c, device_alloc(c, &c->loc.xyz, sizeof(double) * 3 * G));
        CK(c, device_alloc(c, &c->loc.surf, esz * G * c->K + 8));
        CK(c, device_alloc(c, &c->loc.cost, esz * G + 8));
        c->loc.g_cap = (size_t)G;
    }
    return DG_OK;
}

// Half-width (nodes) of the refinement grid of dg_argmax_refine; 0 = none.
static dg_status refine_half(dg_ctx *c, double spacing_m, double window_m, int *half)
{
    *half = 0;
    if (!(spacing_m > 0 && window_m >= spacing_m)) return DG_OK;
    if (!(std::isfinite(spacing_m) && std::isfinite(window_m)))
        return fail(c, DG_EINVAL, "refinement spacing and window must be finite");
    const double h = std::floor(window_m / spacing_m + 0.5);
    if (h > 2000) return fail(c, DG_EINVAL, "refinement grid wider than 4001 nodes");
    *half = (int)h;
    return DG_OK;
}

static dg_status ensure_post(dg_ctx *c, int half, dg_fix **fix_dev, dg_fix **fix_host);
static dg_status step_device_post(dg_ctx *c, const void *cost, double spacing_m, int half, dg_fix *fix_dev,
                                  dg_fix *fix_host, const ArgmaxResult *known);
static dg_status read_fix(dg_ctx *c, const dg_fix *fix_host, dg_fix *out);
static dg_status copy_fix(dg_ctx *c, const dg_fix *fix_host, dg_fix *out);

static dg_status argmax_refine(dg_ctx *c, const void *cost, double spacing_m, double window_m, dg_fix *out,
                               const ArgmaxResult *known)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!cost || !out) return fail(c, DG_EINVAL, "cost and out must not be NULL");
    int half = 0;
    dg_status st = refine_half(c, spacing_m, window_m, &half);
    if (st != DG_OK) return st;
    // the step of a captured graph, uncaptured: the refinement grid is centred
    // on the argmax on the device and one synchronisation reads the fix
    if ((st = ensure_post(c, half, &c->fix_dev_sync, &c->fix_host_sync)) != DG_OK) return st;
    if ((st = step_device_post(c, cost, spacing_m, half, c->fix_dev_sync, c->fix_host_sync, known)) != DG_OK) return st;
    dg_fix f;
    if ((st = read_fix(c, c->fix_host_sync, &f)) != DG_OK) return st;
    *out = f;
    return DG_OK;
}

dg_status dg_argmax_refine(dg_ctx *c, const void *cost, double spacing_m, double window_m, dg_fix *out)
{
    return argmax_refine(c, cost, spacing_m, window_m, out, nullptr);
}

dg_status dg_detect(dg_ctx *c, const void *cost, double threshold, int32_t relative, int32_t radius,
                    int32_t max_peaks, dg_peak *out, int32_t *n_out)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!cost || !out || !n_out) return fail(c, DG_EINVAL, "cost, out and n_out must not be NULL");
    if (radius < 0 || radius > 64) return fail(c, DG_EINVAL, "radius must be in [0, 64]");
    if (max_peaks < 1 || max_peaks > kDetectCap) return fail(c, DG_EINVAL, "max_peaks must be in [1, %d]", kDetectCap);
    if (!std::isfinite(threshold)) return fail(c, DG_EINVAL, "threshold must be finite");
    constexpr int kCap = kDetectCap;
    dg_status st;
    double thr = threshold;
    if (relative) {
        CK(c, cudaStreamSynchronize(c->stream));
        if ((st = check_latched(c)) != DG_OK) return st;
        ArgmaxResult r;
        if ((st = run_argmax(c, cost, c->G, c->gd, &r)) != DG_OK) return st;
        if (r.idx < 0) return fail(c, DG_EINVAL, "the surface holds no finite value");
        thr = threshold * r.val;
    }
    const size_t out_bytes = sizeof(DetectPeak) * kCap + sizeof(int);  // records, then their count
    if (!c->det_cand) CK(c, device_alloc(c, &c->det_cand, sizeof(int64_t) * kCap));
    if (!c->det_out) CK(c, device_alloc(c, &c->det_out, out_bytes));
    if (!c->det_host) CK(c, pinned_alloc(&c->det_host, out_bytes));
    int *const count_d = reinterpret_cast<int *>(c->det_out + max_peaks);  // behind the records asked for
    const DetectPeak *const pk = c->det_host;
    int count = 0;
    for (int round = 0;; ++round) {
        {
            Timed t(c, DG_K_ARGMAX);
            CK(c, launch_detect(cost, c->opt.prec, c->gd, c->gstep, thr, radius, kCap, max_peaks, count_d, c->det_cand,
                                c->det_out, c->stream));
            t.done(2);
        }
        CK(c, cudaMemcpyAsync(c->det_host, c->det_out, sizeof(DetectPeak) * (size_t)max_peaks + sizeof(int),
                              cudaMemcpyDeviceToHost, c->stream));
        CK(c, cudaStreamSynchronize(c->stream));
        if ((st = check_latched(c)) != DG_OK) return st;
        count = *reinterpret_cast<const int *>(c->det_host + max_peaks);
        if (count <= kCap) break;
        // More peaks pass than the sort holds: it ordered kCap of them (an
        // arbitrary subset), so at least max_peaks peaks reach its
        // max_peaks-th value, and so does every one of the max_peaks largest.
        // That value is the next threshold; far fewer peaks pass it.
        const double next = pk[(size_t)max_peaks - 1].value;
        if (!(next > thr) || round >= 8)
            return fail(c, DG_EUNSUPPORTED, "%d peaks of equal value pass the detection test (max %d); raise the "
                        "threshold", count, kCap);
        thr = next;
    }
    const int n = std::min(count, (int)max_peaks);
    for (int k = 0; k < n; ++k) {
        out[k].index = pk[k].index;
        out[k].i = pk[k].i;
        out[k].j = pk[k].j;
        out[k].lat_deg = pk[k].lat_rad * (180.0 / kPi);
        out[k].lon_deg = pk[k].lon_rad * (180.0 / kPi);
        out[k].value = pk[k].value;
    }
    *n_out = n;
    return DG_OK;
}

// ---------------------------------------------------------------------------
// Whole steps as CUDA graphs
// ---------------------------------------------------------------------------

// Buffers of a step after its surface (allocated outside any capture).
static dg_status ensure_post(dg_ctx *c, int half, dg_fix **fix_dev, dg_fix **fix_host)
{
    const int n = 2 * half + 1;
    const int64_t Gl = half > 0 ? (int64_t)n * n : 0;
    dg_status st;
    if ((st = ensure(c, &c->amax_tmp, &c->amax_tmp_bytes, argmax_tmp_bytes(std::max<int64_t>(c->G, Gl)))) != DG_OK)
        return st;
    if (half > 0 && (st = ensure_local(c, Gl)) != DG_OK) return st;
    if (!c->amax_fine) CK(c, device_alloc(c, &c->amax_fine, sizeof(ArgmaxResult)));
    if (!*fix_dev) CK(c, device_alloc(c, fix_dev, sizeof(dg_fix)));
    if (!*fix_host) CK(c, pinned_alloc(fix_host, sizeof(dg_fix)));
    return DG_OK;
}

// Buffers a device-only step needs (allocated outside any capture).
static dg_status prepare_step(dg_ctx *c, int half)
{
    for (int k = 0; k < c->K; ++k)
        if (!c->steps[k].loaded) return fail(c, DG_ESTATE, "snapshot %d has not been loaded", k);
    dg_status st = ensure_surf(c);
    if (st != DG_OK) return st;
    if ((st = ensure_post(c, half, &c->fix_dev, &c->fix_host)) != DG_OK) return st;
    return push_steps(c);
}

// One step on the device only: the surface into cost, its argmax, the
// refinement grid centred on it (built on the device), the refinement
// surface and argmax, and the fix record copied to the pinned fix_host. No
// host synchronisation and no allocation (prepare_step ran before).
static dg_status step_device(dg_ctx *c, void *cost, double spacing_m, int half)
{
    dg_status st = run_surface(c, c->gd, c->xyz, c->G, c->surf, cost, false);
    if (st != DG_OK) return st;
    return step_device_post(c, cost, spacing_m, half, c->fix_dev, c->fix_host, nullptr);
}

// The rest of a step once the surface is enqueued: its argmax (unless its record
// is on the device: known), the refinement, the fix record.
static dg_status step_device_post(dg_ctx *c, const void *cost, double spacing_m, int half, dg_fix *fix_dev,
                                  dg_fix *fix_host, const ArgmaxResult *known)
{
    dg_status st = DG_OK;
    if (known && half > 0) {  // the surface's record is on the device already
        CK(c, cudaMemcpyAsync(c->amax_res, known, sizeof(ArgmaxResult), cudaMemcpyDeviceToDevice, c->stream));
    } else {
        Timed t(c, DG_K_ARGMAX);
        int nl = 0;
        CK(c, launch_argmax(cost, c->G, c->opt.prec, c->gd, c->gstep, c->amax_tmp, c->amax_res, &nl, c->stream, nullptr,
                            nullptr, 1, FixOut{half > 0 ? nullptr : fix_dev, nullptr, c->gd, 0}));
        t.done(nl);
    }
    const int n = 2 * half + 1;
    if (half > 0) {
        dg_grid lg;
        lg.lat0_deg = c->grid.lat0_deg;  // replaced on the device by the argmax node
        lg.lon0_deg = c->grid.lon0_deg;
        lg.dlat_m = lg.dlon_m = spacing_m;
        lg.nlat = lg.nlon = n;
        const GridDev lgd = make_griddev(lg, 0, n);
        const int64_t Gl = (int64_t)n * n;
        {
            Timed t(c, DG_K_REFINE);
            CK(c, launch_grid_ecef(lgd, c->loc.xyz, c->stream, c->amax_res, nullptr, 1, c->gstep + 1));
            t.done(1);
        }
        st = run_surface(c, lgd, c->loc.xyz, Gl, c->loc.surf, c->loc.cost, true);
        if (st != DG_OK) return st;
        {
            Timed t(c, DG_K_ARGMAX);
            int nl = 0;
            CK(c, launch_argmax(c->loc.cost, Gl, c->opt.prec, lgd, c->gstep + 1, c->amax_tmp, c->amax_fine, &nl, c->stream,
                                c->amax_res, nullptr, 1, FixOut{fix_dev, c->amax_res, c->gd, n}));
            t.done(nl);
        }
    }
    CK(c, cudaMemcpyAsync(fix_host, fix_dev, sizeof(dg_fix), cudaMemcpyDeviceToHost, c->stream));
    return DG_OK;
}

static dg_status read_fix(dg_ctx *c, const dg_fix *fix_host, dg_fix *out)
{
    CK(c, cudaStreamSynchronize(c->stream));
    const dg_status st = check_latched(c);
    return st != DG_OK ? st : copy_fix(c, fix_host, out);
}

// The fix of a step that has been waited for.
static dg_status copy_fix(dg_ctx *c, const dg_fix *fix_host, dg_fix *out)
{
    if (fix_host->index < 0) return fail(c, DG_EINVAL, "the surface holds no finite value");
    if (fix_host->refine_n > 0 && fix_host->ri < 0)
        return fail(c, DG_EINVAL, "the refinement surface holds no finite value");
    *out = *fix_host;
    return DG_OK;
}

// Capture one step of each context as a branch of one graph: forked from and
// joined to `stream`. Timing is off inside the capture.
// The shared contraction rounds of a batch (dg_batch_capture): round r runs,
// in one persistent launch, the contraction of the r-th snapshot batch of
// every context that has one; each context plans and combines its batch on
// its own stream around it.
struct TcRounds {
    std::vector<std::vector<int>> ctx;  // per round: the contexts taking part
    std::vector<int> job_off;           // per round: its first job in jobs
    std::vector<int> tile_off;          // per round: its prefix sums in job_tiles
    TcJob *jobs = nullptr;              // device, every round's jobs in order
    int *job_tiles = nullptr;           // device, per round n_r + 1 tile prefix sums
    int fmt = 0, contract = 0;
    unsigned wait_polls = 0;
};

// Every context on the tensor-core CDFT path (lag or row tiles), one capture
// format and one contraction arithmetic across all of them: the batch's
// contractions can share launches. The contexts have run one uncaptured
// step, so their layouts and buffers exist. Builds the job tables on the
// device (synchronously, before any capture).
static dg_status tc_rounds(dg_ctx *const *ctxs, int n, TcRounds &R, bool &ok)
{
    ok = false;
    if (n < 2) return DG_OK;
    const int fmt = ctxs[0]->steps[0].fmt, contract = ctxs[0]->opt.contract;
    size_t rounds = 0;
    for (int i = 0; i < n; ++i) {
        dg_ctx *c = ctxs[i];
        if (c->opt.algo != DG_ALGO_CDFT || c->opt.contract == DG_CONTRACT_FP32 || c->opt.tiles == DG_TILES_HANKEL ||
            c->opt.contract != contract || !c->cd.main_run.L || c->last_map)
            return DG_OK;
        for (int k = 0; k < c->K; ++k)
            if (c->steps[k].fmt != fmt) return DG_OK;
        rounds = std::max(rounds, c->cd.main_run.L->batches.size());
    }
    std::vector<TcJob> jobs;
    R.ctx.assign(rounds, {});
    for (size_t r = 0; r < rounds; ++r) {
        R.job_off.push_back((int)jobs.size());
        R.tile_off.push_back((int)(jobs.size() + r));
        for (int i = 0; i < n; ++i) {
            dg_ctx *c = ctxs[i];
            if (r >= c->cd.main_run.L->batches.size()) continue;
            CdftBatch a{};
            cdft_args(c, c->cd.main_run, r, a);
            jobs.push_back(tc_job(a, a.btab));
            R.ctx[r].push_back(i);
        }
    }
    dg_ctx *c0 = ctxs[0];
    auto table = [](auto **p, size_t bytes) {  // NULL where it fails (tc_rounds_free)
        const cudaError_t e = cudaMalloc((void **)p, bytes);
        if (e != cudaSuccess) {
            *p = nullptr;
            cudaGetLastError();
        }
        return e;
    };
    CK(c0, table(&R.jobs, sizeof(TcJob) * jobs.size()));
    CK(c0, table(&R.job_tiles, sizeof(int) * (jobs.size() + rounds)));
    CK(c0, cudaMemcpy(R.jobs, jobs.data(), sizeof(TcJob) * jobs.size(), cudaMemcpyHostToDevice));
    R.fmt = fmt;
    R.contract = contract;
    R.wait_polls = g_tc_wait_polls.load(std::memory_order_relaxed);
    ok = true;
    return DG_OK;
}

static void tc_rounds_free(TcRounds &R)
{
    if (R.jobs) cudaFree(R.jobs);
    if (R.job_tiles) cudaFree(R.job_tiles);
    R.jobs = nullptr;
    R.job_tiles = nullptr;
}

// The surfaces of a batch's contexts with shared contraction rounds (inside
// a capture): setup, then per round every context's plan, one launch, every
// context's combine; then each context's accumulation. Returns the shared
// launches in *shared.
static dg_status shared_surfaces(dg_ctx *const *ctxs, int n, void *const *costs, const TcRounds &R,
                                 cudaStream_t stream, int64_t *shared)
{
    dg_ctx *c0 = ctxs[0];
    std::vector<CdftRun> runs((size_t)n);
    for (int i = 0; i < n; ++i) {
        dg_ctx *c = ctxs[i];
        CdftRun &r = runs[(size_t)i];
        r.gd = c->gd;
        r.xyz = c->xyz;
        r.G = c->G;
        r.surf = c->surf;
        r.out = costs[i];
        r.refine = false;
        dg_status st = cdft_setup(c, r);
        if (st != DG_OK) return st;
    }
    std::vector<cudaEvent_t> evs;
    auto event = [&](cudaEvent_t *e) {
        const cudaError_t x = cudaEventCreateWithFlags(e, cudaEventDisableTiming);
        if (x == cudaSuccess) evs.push_back(*e);
        return x;
    };
    dg_status st = DG_OK;
    cudaError_t e = cudaSuccess;
    for (size_t rd = 0; rd < R.ctx.size() && st == DG_OK && e == cudaSuccess; ++rd) {
        const std::vector<int> &part = R.ctx[rd];
        for (int i : part) {
            dg_ctx *c = ctxs[i];
            CdftBatch a{};
            cdft_args(c, runs[(size_t)i], rd, a);
            if ((st = cdft_plan(c, runs[(size_t)i], a, rd)) != DG_OK) break;
            if ((st = cdft_contract(c, runs[(size_t)i], a, rd, true)) != DG_OK) break;
            cudaEvent_t ev;
            if ((e = event(&ev)) != cudaSuccess || (e = cudaEventRecord(ev, c->stream)) != cudaSuccess ||
                (e = cudaStreamWaitEvent(stream, ev, 0)) != cudaSuccess)
                break;
        }
        if (st != DG_OK || e != cudaSuccess) break;
        const int nr = (int)part.size();
        TcJob *jobs = R.jobs + R.job_off[rd];
        int *tiles = R.job_tiles + R.tile_off[rd];
        if ((e = launch_tc_job_tiles(jobs, nr, tiles, stream)) != cudaSuccess) break;
        if ((e = launch_cdft_contract_jobs(jobs, nr, tiles, c0->sm_count, R.fmt, R.contract, R.wait_polls, stream)) !=
            cudaSuccess)
            break;
        *shared += 2;
        cudaEvent_t done;
        if ((e = event(&done)) != cudaSuccess || (e = cudaEventRecord(done, stream)) != cudaSuccess) break;
        for (int i : part) {
            dg_ctx *c = ctxs[i];
            if ((e = cudaStreamWaitEvent(c->stream, done, 0)) != cudaSuccess) break;
            CdftBatch a{};
            cdft_args(c, runs[(size_t)i], rd, a);
            if ((st = cdft_combine(c, runs[(size_t)i], a, rd)) != DG_OK) break;
        }
    }
    for (int i = 0; i < n && st == DG_OK && e == cudaSuccess; ++i) st = cdft_finish(ctxs[i], runs[(size_t)i]);
    for (auto &x : evs) cudaEventDestroy(x);
    if (st != DG_OK) return st;
    if (e != cudaSuccess) return fail(c0, DG_ECUDA, "shared contraction rounds: %s", cudaGetErrorString(e));
    return DG_OK;
}

static dg_status capture_steps(dg_ctx *const *ctxs, int n, void *const *costs, double spacing_m, const int *half,
                               cudaStream_t stream, cudaGraphExec_t *exec, int64_t *launches,
                               const TcRounds *rounds = nullptr)
{
    dg_ctx *c0 = ctxs[0];
    cudaEvent_t fork = nullptr;
    std::vector<cudaEvent_t> join((size_t)n, nullptr);
    CK(c0, cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
    for (auto &e : join) CK(c0, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    std::vector<int> timing((size_t)n);
    std::vector<int64_t> l0((size_t)n);
    dg_status st = DG_OK;
    int64_t shared = 0;
    cudaError_t e = cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) e = cudaEventRecord(fork, stream);
    for (int i = 0; i < n; ++i) {
        timing[i] = ctxs[i]->opt.timing;
        ctxs[i]->opt.timing = 0;
        l0[i] = ctxs[i]->launches;
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ctxs[i]->stream, fork, 0);
    }
    if (rounds && e == cudaSuccess) st = shared_surfaces(ctxs, n, costs, *rounds, stream, &shared);
    for (int i = 0; i < n && e == cudaSuccess && st == DG_OK; ++i) {
        dg_ctx *c = ctxs[i];
        st = rounds ? step_device_post(c, costs[i], spacing_m, half[i], c->fix_dev, c->fix_host, nullptr)
                    : step_device(c, costs[i], spacing_m, half[i]);
        if (st == DG_OK) e = cudaEventRecord(join[i], c->stream);
        if (e == cudaSuccess && st == DG_OK) e = cudaStreamWaitEvent(stream, join[i], 0);
    }
    for (int i = 0; i < n; ++i) ctxs[i]->opt.timing = timing[i];
    cudaGraph_t g = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(stream, &g);
    if (e == cudaSuccess) e = e2;
    int64_t total = shared;
    for (int i = 0; i < n; ++i) {
        const int64_t d = ctxs[i]->launches - l0[i];
        total += d;
        ctxs[i]->launches = l0[i];  // counted again at each replay
    }
    if (st == DG_OK && e == cudaSuccess) e = cudaGraphInstantiate(exec, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaEventDestroy(fork);
    for (auto &j : join) cudaEventDestroy(j);
    if (st != DG_OK) return st;
    if (e != cudaSuccess) return fail(c0, DG_ECUDA, "graph capture: %s", cudaGetErrorString(e));
    *launches = total;
    return DG_OK;
}

dg_status dg_graph_capture(dg_ctx *c, void *cost, double spacing_m, double window_m)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!cost) return fail(c, DG_EINVAL, "cost is NULL");
    if (!c->stream || c->stream == cudaStreamLegacy || c->stream == cudaStreamPerThread)
        return fail(c, DG_EUNSUPPORTED, "graph capture needs a context created on a non-default stream");
    int half = 0;
    dg_status st = refine_half(c, spacing_m, window_m, &half);
    if (st != DG_OK) return st;
    if (c->graph) {
        cudaGraphExecDestroy(c->graph);
        c->graph = nullptr;
    }
    if ((st = give_back(c)) != DG_OK) return st;
    // one uncaptured step allocates and plans everything; then the capture
    if ((st = prepare_step(c, half)) != DG_OK) return st;
    if ((st = step_device(c, cost, spacing_m, half)) != DG_OK) return st;
    dg_fix f;
    if ((st = read_fix(c, c->fix_host, &f)) != DG_OK) return st;
    dg_ctx *const cs[1] = {c};
    void *const costs[1] = {cost};
    if ((st = capture_steps(cs, 1, costs, spacing_m, &half, c->stream, &c->graph, &c->graph_launches)) != DG_OK)
        return st;
    c->graph_gen = c->steps_gen;
    return DG_OK;
}

dg_status dg_graph_launch(dg_ctx *c)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!c->graph) return fail(c, DG_ESTATE, "no graph has been captured");
    if (c->graph_gen != c->steps_gen || c->steps_dirty)
        return fail(c, DG_ESTATE, "a capture changed format, length or buffer since the graph was captured");
    CK(c, cudaGraphLaunch(c->graph, c->stream));
    c->launches += c->graph_launches;
    return DG_OK;
}

dg_status dg_graph_fix(dg_ctx *c, dg_fix *out)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!out) return fail(c, DG_EINVAL, "out is NULL");
    if (!c->fix_host) return fail(c, DG_ESTATE, "no step has run");
    return read_fix(c, c->fix_host, out);
}

}  // extern "C" (reopened below)

struct dg_batch {
    std::vector<dg_ctx *> ctxs;
    std::vector<uint64_t> gens;
    std::vector<cudaEvent_t> ready;  // work queued on each context's stream
    std::vector<std::shared_ptr<BatchHold>> holds;  // of the contexts
    cudaEvent_t last = nullptr;      // behind the latest replay
    cudaStream_t stream = nullptr;
    cudaGraphExec_t graph = nullptr;
    int64_t launches = 0;
    std::string err;
    TcRounds rounds;       // shared contraction rounds (none: per-context launches)
    bool shared = false;
};

extern "C" {

dg_status dg_batch_capture(dg_ctx *const *ctxs, int32_t n, void *const *costs, double spacing_m, double window_m,
                           void *stream, dg_batch **out)
{
    if (!out) return fail(nullptr, DG_EINVAL, "out is NULL");
    *out = nullptr;
    if (!ctxs || !costs || n < 1) return fail(nullptr, DG_EINVAL, "ctxs and costs must hold n >= 1 entries");
    cudaStream_t s = (cudaStream_t)stream;
    if (!s || s == cudaStreamLegacy || s == cudaStreamPerThread)
        return fail(nullptr, DG_EUNSUPPORTED, "graph capture needs a non-default stream");
    std::vector<int> half((size_t)n);
    double fill = 0.0;
    for (int i = 0; i < n; ++i)
        if (ctxs[i]) fill += grid_tiles(ctxs[i], ctxs[i]->gd);
    struct Filled {  // the steps below are planned for the whole batch's work
        dg_ctx *const *ctxs;
        int n;
        void set(double f)
        {
            for (int i = 0; i < n; ++i)
                if (ctxs[i]) ctxs[i]->cd.fill = f;
        }
        ~Filled() { set(0.0); }
    } filled{ctxs, n};
    filled.set(fill);
    for (int i = 0; i < n; ++i) {
        dg_ctx *c = ctxs[i];
        if (!c || !costs[i]) return fail(nullptr, DG_EINVAL, "context or cost %d is NULL", i);
        if (c->device != ctxs[0]->device) return fail(nullptr, DG_EINVAL, "the contexts must share one device");
        if (!c->stream || c->stream == cudaStreamLegacy || c->stream == cudaStreamPerThread)
            return fail(nullptr, DG_EUNSUPPORTED, "context %d is on a default stream", i);
        c->err.clear();
        dg_status st = refine_half(c, spacing_m, window_m, &half[i]);
        if (st == DG_OK) st = prepare_step(c, half[i]);
        if (st == DG_OK) st = step_device(c, costs[i], spacing_m, half[i]);
        dg_fix f;
        if (st == DG_OK) st = read_fix(c, c->fix_host, &f);
        if (st != DG_OK) return fail(nullptr, st, "context %d: %s", i, c->err.c_str());
    }
    dg_batch *b = new (std::nothrow) dg_batch();
    if (!b) return fail(nullptr, DG_ENOMEM, "host allocation failed");
    b->ctxs.assign(ctxs, ctxs + n);
    for (int i = 0; i < n; ++i) b->gens.push_back(ctxs[i]->steps_gen);
    b->ready.assign((size_t)n, nullptr);
    bool events = cudaEventCreateWithFlags(&b->last, cudaEventDisableTiming) == cudaSuccess;
    for (auto &e : b->ready) events = events && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    if (!events) {
        dg_batch_destroy(b);
        return fail(nullptr, DG_ECUDA, "event creation failed");
    }
    b->stream = s;
    dg_status st = tc_rounds(ctxs, n, b->rounds, b->shared);
    if (st == DG_OK)
        st = capture_steps(ctxs, n, costs, spacing_m, half.data(), s, &b->graph, &b->launches,
                           b->shared ? &b->rounds : nullptr);
    if (st != DG_OK) {
        const std::string m = ctxs[0]->err;
        dg_batch_destroy(b);
        return fail(nullptr, st, "%s", m.c_str());
    }
    for (int i = 0; i < n; ++i) {
        auto h = std::make_shared<BatchHold>();
        h->last = b->last;
        h->fill = fill;
        h->gen = ctxs[i]->steps_gen;
        b->holds.push_back(h);
        ctxs[i]->holds.push_back(h);
    }
    *out = b;
    return DG_OK;
}

dg_status dg_batch_launch(dg_batch *b)
{
    if (!b || !b->graph) return fail(nullptr, DG_EINVAL, "no batch graph");
    for (size_t i = 0; i < b->ctxs.size(); ++i)
        if (b->ctxs[i]->steps_gen != b->gens[i] || b->ctxs[i]->steps_dirty)
            return fail(nullptr, DG_ESTATE, "context %zu changed a capture's format, length or buffer", i);
    // the steps read what was queued on the contexts' own streams (capture
    // loads): order the launch after it
    for (size_t i = 0; i < b->ctxs.size(); ++i) {
        cudaError_t e = cudaEventRecord(b->ready[i], b->ctxs[i]->stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->ready[i], 0);
        if (e != cudaSuccess) return fail(nullptr, DG_ECUDA, "ordering the launch: %s", cudaGetErrorString(e));
    }
    const cudaError_t e = cudaGraphLaunch(b->graph, b->stream);
    if (e != cudaSuccess) return fail(nullptr, DG_ECUDA, "cudaGraphLaunch: %s", cudaGetErrorString(e));
    const cudaError_t r = cudaEventRecord(b->last, b->stream);
    if (r != cudaSuccess) return fail(nullptr, DG_ECUDA, "cudaEventRecord: %s", cudaGetErrorString(r));
    return DG_OK;
}

dg_status dg_batch_fixes(dg_batch *b, dg_fix *out)
{
    if (!b || !out) return fail(nullptr, DG_EINVAL, "batch and out must not be NULL");
    const cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return fail(nullptr, DG_ECUDA, "cudaStreamSynchronize: %s", cudaGetErrorString(e));
    dg_status worst = DG_OK;
    for (size_t i = 0; i < b->ctxs.size(); ++i) {
        dg_status st = read_fix(b->ctxs[i], b->ctxs[i]->fix_host, &out[i]);
        if (st != DG_OK) {
            std::memset(&out[i], 0, sizeof(dg_fix));
            out[i].index = -1;
            if (worst == DG_OK) {
                worst = st;
                fail(nullptr, st, "context %zu: %s", i, b->ctxs[i]->err.c_str());
            }
        }
    }
    return worst;
}

int64_t dg_batch_launch_count(const dg_batch *b) { return b ? b->launches : -1; }

dg_status dg_batch_destroy(dg_batch *b)
{
    if (!b) return DG_OK;
    // the contexts may free what its replays read once they are done
    if (b->last) cudaEventSynchronize(b->last);
    for (auto &h : b->holds) h->alive = false;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->last) cudaEventDestroy(b->last);
    for (auto &e : b->ready)
        if (e) cudaEventDestroy(e);
    tc_rounds_free(b->rounds);
    delete b;
    return DG_OK;
}

int32_t dg_batch_rounds(const dg_batch *b) { return b && b->shared ? (int32_t)b->rounds.ctx.size() : 0; }

// ---------------------------------------------------------------------------
// Autotuning of the CDFT launch shape
// ---------------------------------------------------------------------------
namespace {
std::mutex g_tune_mutex;
// a tuned shape: chunk and tiles (CDFT) or rows (DIRECT)
struct TuneShape {
    int chunk = 0, tiles = 0, rows = 0;
};
std::map<std::string, TuneShape> g_tune_cache;

std::string tune_key(const dg_ctx *c)
{
    std::string k = std::to_string(c->G) + "/" + std::to_string(c->gd.nlon) + "/" + std::to_string(c->K) + "/" +
                    std::to_string(c->opt.algo) + "/" + std::to_string(c->opt.prec) + "/" +
                    std::to_string(c->opt.delay) + "/" + std::to_string(c->opt.contract) + "/" +
                    std::to_string(c->opt.acc) + "/" + std::to_string(c->fs);
    for (const auto &st : c->steps) k += "/" + std::to_string(st.n) + ":" + std::to_string(st.fmt);
    return k;
}
}  // namespace

dg_status dg_autotune(dg_ctx *c, void *cost, int32_t reps, dg_tuning *out)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!cost || !out) return fail(c, DG_EINVAL, "cost and out must not be NULL");
    if (reps < 1 || reps > 100) return fail(c, DG_EINVAL, "reps must be in [1, 100]");
    for (int k = 0; k < c->K; ++k)
        if (!c->steps[k].loaded) return fail(c, DG_ESTATE, "snapshot %d has not been loaded", k);
    std::memset(out, 0, sizeof *out);
    const bool cdft = c->opt.algo == DG_ALGO_CDFT;
    auto apply = [&](const TuneShape &t) {
        if (cdft) {
            c->opt.chunk = t.chunk;
            c->opt.tiles = t.tiles;
            out->chunk = t.chunk;
            out->tiles = t.tiles;
        } else {
            c->opt.rows = t.rows;
            out->rows = t.rows;
        }
    };
    const std::string key = tune_key(c);
    {
        std::lock_guard<std::mutex> lk(g_tune_mutex);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            apply(it->second);
            out->cached = 1;
            return DG_OK;
        }
    }
    std::vector<TuneShape> shapes;
    if (cdft) {
        // admissible chunks: the automatic rule's bound on the estimated spacing
        std::vector<double> &span = c->cd.main_span;
        if (span.size() != (size_t)c->K || c->cd.main_lags.size() != (size_t)c->K)
            fdoa_spans(c, c->gd, span, &c->cd.main_lags);
        double dmax = 0.0;
        int64_t nmin = INT64_MAX;
        for (int k = 0; k < c->K; ++k) {
            dmax = std::max(dmax, span[k] * (1.0 + 1e-5) / kCdftBinSpan);
            nmin = std::min<int64_t>(nmin, c->steps[k].n);
        }
        const bool tc = c->opt.contract != DG_CONTRACT_FP32;
        std::vector<int> chunks;
        for (int m = 256; m <= (tc ? kCdftAutoMaxChunkTc : kCdftAutoMaxChunk); m *= 2)
            if (1.1 * m * dmax <= kCdftMDelta && (m <= kCdftAutoMaxChunk || m <= nmin)) chunks.push_back(m);
        if (chunks.empty()) chunks.push_back(auto_chunk(c, span, c->cd.main_lags, 0, c->K, tc));
        std::vector<int> tiles = {DG_TILES_ROWS};
        if (tc) {
            tiles.push_back(DG_TILES_LAGS);
            tiles.push_back(DG_TILES_HANKEL);
        }
        for (int m : chunks)
            for (int t : tiles) {
                if (t == DG_TILES_HANKEL && m > kLagTileMaxChunk) continue;
                if (t == DG_TILES_LAGS && m > kLagTileMaxChunk && m % kLagTileMaxChunk != 0) continue;
                TuneShape sh;
                sh.chunk = m;
                sh.tiles = t;
                shapes.push_back(sh);
            }
    } else {
        // grid rows per thread: candidates per CTA and the CTA's lag span
        // (16 rows of 4-tap interpolation weights spill registers: not tried)
        const std::vector<int> rows = c->opt.prec == DG_PREC_FP64         ? std::vector<int>{2, 4}
                                      : c->opt.delay == DG_DELAY_INTEGER ? std::vector<int>{4, 8, 16}
                                                                         : std::vector<int>{4, 8};
        for (int r : rows) {
            TuneShape sh;
            sh.rows = r;
            shapes.push_back(sh);
        }
    }
    const dg_options saved = c->opt;
    const size_t esz = c->opt.prec == DG_PREC_FP64 ? 8 : 4;
    dg_status st = ensure(c, &c->surf, &c->surf_bytes, esz * (size_t)c->G * c->K);
    if (st != DG_OK) return st;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    CK(c, cudaEventCreate(&e0));
    CK(c, cudaEventCreate(&e1));
    double best = 1e300;
    TuneShape best_sh = shapes[0];
    c->opt.timing = 0;  // restored with the saved options
    for (const TuneShape &sh : shapes) {
        if (cdft) {
            c->opt.chunk = sh.chunk;
            c->opt.tiles = sh.tiles;
        } else {
            c->opt.rows = sh.rows;
        }
        std::vector<float> ms;
        for (int r = 0; r <= reps && st == DG_OK; ++r) {
            if (r > 0 && cudaEventRecord(e0, c->stream) != cudaSuccess) st = DG_ECUDA;
            if (st == DG_OK) st = run_surface(c, c->gd, c->xyz, c->G, c->surf, cost, false);
            if (st == DG_OK && r > 0 && cudaEventRecord(e1, c->stream) != cudaSuccess) st = DG_ECUDA;
            if (st == DG_OK && cudaStreamSynchronize(c->stream) != cudaSuccess) st = DG_ECUDA;
            if (st == DG_OK) st = check_latched(c);
            float x = 0.f;
            if (st == DG_OK && r > 0) {
                cudaEventElapsedTime(&x, e0, e1);
                ms.push_back(x);
            }
        }
        if (st != DG_OK) break;
        std::sort(ms.begin(), ms.end());
        const double med = ms[ms.size() / 2];
        ++out->tried;
        if (med < best) {
            best = med;
            best_sh = sh;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->opt = saved;
    if (st != DG_OK) {
        if (c->err.empty()) fail(c, st, "a timed surface failed");
        return st;
    }
    apply(best_sh);
    out->ms = best;
    std::lock_guard<std::mutex> lk(g_tune_mutex);
    g_tune_cache[key] = best_sh;
    return DG_OK;
}

dg_status dg_grid_ecef(dg_ctx *c, double *xyz_out)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!xyz_out) return fail(c, DG_EINVAL, "xyz_out is NULL");
    if (need_nodes(c) != DG_OK) return DG_ENOMEM;
    CK(c, cudaMemcpyAsync(xyz_out, c->xyz, sizeof(double) * 3 * (size_t)c->G, cudaMemcpyDeviceToDevice,
                          c->stream));
    return DG_OK;
}

dg_status dg_step_geometry(dg_ctx *c, int32_t step, int32_t *lag, double *D, double *nu)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (step < 0 || step >= c->K) return fail(c, DG_EINVAL, "step %d outside [0, %d)", step, c->K);
    if (need_nodes(c) != DG_OK) return DG_ENOMEM;
    {
        Timed t(c, DG_K_GRID);
        CK(c, launch_step_geometry(c->gd, c->xyz, c->eph + 12 * (size_t)step, c->fs, c->lambda,
                                   c->opt.delay, lag, D, nu, c->stream));
        t.done(1);
    }
    return DG_OK;
}

dg_status dg_kernel_time(dg_ctx *c, int32_t cls, double *ms, int64_t *launches)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (cls < 0 || cls >= DG_K_NCLASS) return fail(c, DG_EINVAL, "unknown kernel class %d", cls);
    CK(c, cudaStreamSynchronize(c->stream));
    for (auto &t : c->pending) {
        float v = 0;
        cudaEventElapsedTime(&v, t.a, t.b);
        c->ms[t.cls] += v;
        cudaEventDestroy(t.a);
        cudaEventDestroy(t.b);
    }
    c->pending.clear();
    if (ms) *ms = c->ms[cls];
    if (launches) *launches = c->nl[cls];
    return DG_OK;
}

dg_status dg_reset_counters(dg_ctx *c)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    CK(c, cudaStreamSynchronize(c->stream));
    for (auto &t : c->pending) {
        cudaEventDestroy(t.a);
        cudaEventDestroy(t.b);
    }
    c->pending.clear();
    for (int i = 0; i < DG_K_NCLASS; ++i) {
        c->ms[i] = 0;
        c->nl[i] = 0;
    }
    c->launches = 0;
    return DG_OK;
}

int64_t dg_launch_count(const dg_ctx *c) { return c ? c->launches : -1; }

dg_status dg_cdft_chunks(const dg_ctx *c, int32_t *min_chunk, int32_t *max_chunk)
{
    if (!c) return DG_EINVAL;
    if (c->cd_chunk_max < 0) {  // the last surfaces were regions': the grid the context was left on
        dg_ctx *m = const_cast<dg_ctx *>(c);
        if (!map_chunks(m, &m->cd_chunk_min, &m->cd_chunk_max)) m->cd_chunk_min = m->cd_chunk_max = 0;
    }
    const bool any = c->cd_chunk_max > 0;
    if (min_chunk) *min_chunk = any ? c->cd_chunk_min : 0;
    if (max_chunk) *max_chunk = any ? c->cd_chunk_max : 0;
    return DG_OK;
}

dg_status dg_cdft_work(const dg_ctx *c, int64_t *bucket_chunks, int64_t *candidate_chunks)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    unsigned long long w[2] = {0, 0};
    if (c->last_map) {  // (lag, block) pairs correlated, candidates looked up
        w[0] = (unsigned long long)c->mp.rows;
        w[1] = (unsigned long long)c->G * c->K;
    } else if (c->cd.work) {  // counted on the device by the plan: wait for the stream
        if (cudaMemcpyAsync(w, c->cd.work, sizeof w, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess)
            return fail(nullptr, DG_ECUDA, "reading the CDFT work counters failed");
    }
    if (bucket_chunks) *bucket_chunks = (int64_t)w[0];
    if (candidate_chunks) *candidate_chunks = (int64_t)w[1];
    return DG_OK;
}

dg_status dg_destroy(dg_ctx *c)
{
    if (!c) return DG_OK;
    cudaStream_t s = c->stream;
    for (auto &t : c->pending) {
        cudaEventDestroy(t.a);
        cudaEventDestroy(t.b);
    }
    auto fr = [&](void *p) {
        if (p) cudaFreeAsync(p, s);
    };
    for (void *p : c->retired) fr(p);
    for (const CdftLayout &L : c->cd.kept) {
        fr(L.bbase);
        fr(L.gbase);
    }
    fr(c->xyz);
    fr(c->gstep);
    fr(c->reg_steps);
    fr(c->eph);
    fr(c->steps_d);
    fr(c->surf);
    fr(c->amax_tmp);
    fr(c->amax_res);
    fr(c->amax_fine);
    fr(c->fix_dev);
    fr(c->fix_dev_sync);
    if (c->graph) cudaGraphExecDestroy(c->graph);
    fr(c->err_d);
    fr(c->det_cand);
    fr(c->det_out);
    fr(c->loc.xyz);
    fr(c->loc.surf);
    fr(c->loc.cost);
    fr(c->cd.lr);
    fr(c->reg_res);
    fr(c->mb.snap);
    fr(c->mb.tw);
    fr(c->mb.T);
    fr(c->mb.F2);
    fr(c->mb.U);
    fr(c->mb.X);
    fr(c->mb.phase);
    fr(c->mb.bad);
    fr(c->reg_xyz);
    fr(c->reg_grids);
    fr(c->mr.snap);
    fr(c->mr.U);
    fr(c->mr.X);
    fr(c->mr.bad);
    fr(c->mb.fit);
    fr(c->mb.coef);
    fr(c->co.lag);
    fr(c->co.nu);
    fr(c->co.lmm);
    fr(c->co.nmm);
    fr(c->co.st);
    fr(c->co.P);
    fr(c->co.tw);
    fr(c->co.F2);
    fr(c->co.pool);
    fr(c->co.turn);
    fr(c->co.snap);
    fr(c->co.bad);
    fr(c->co.A);
    fr(c->co.part);
    fr(c->cd.part);
    fr(c->cd.dmain_layout.bbase);
    fr(c->cd.dmain_layout.gbase);
    fr(c->cd.dloc_layout.bbase);
    fr(c->cd.dloc_layout.gbase);
    fr(c->cd.main_layout.bbase);
    fr(c->cd.main_layout.gbase);
    fr(c->cd.loc_layout.bbase);
    fr(c->cd.loc_layout.gbase);
    fr(c->cd.layout);
    fr(c->cd.Mcs);
    fr(c->cd.work);
    fr(c->cd.candL);
    fr(c->cd.order);
    fr(c->cd.nuS);
    fr(c->cd.g2b);
    fr(c->cd.candNu);
    fr(c->cd.candMu);
    fr(c->cd.muS);
    fr(c->cd.need);
    fr(c->cd.xyzf);
    fr(c->cd.ephf);
    fr(c->cd.count);
    fr(c->cd.offs);
    fr(c->cd.subcnt);
    fr(c->cd.nur);
    fr(c->cd.nubase);
    fr(c->cd.delta);
    fr(c->cd.V);
    fr(c->cd.W);
    fr(c->cd.tbase);
    fr(c->cd.hbase);
    fr(c->cd.btab);
    for (auto &st : c->steps) {
        fr(st.y1);
        fr(st.y2);
    }
    cudaError_t e = cudaStreamSynchronize(s);
    if (c->amax_host) cudaFreeHost(c->amax_host);
    if (c->reg_host) cudaFreeHost(c->reg_host);
    if (c->det_host) cudaFreeHost(c->det_host);
    if (c->fix_host) cudaFreeHost(c->fix_host);
    if (c->fix_host_sync) cudaFreeHost(c->fix_host_sync);
    if (c->err_h) cudaFreeHost(c->err_h);
    delete c;
    if (e != cudaSuccess) return fail(nullptr, DG_ECUDA, "dg_destroy: %s", cudaGetErrorString(e));
    return DG_OK;
}

// ---------------------------------------------------------------------------
// Coarse delay-Doppler maps back-projected onto the grid's cells.
// ---------------------------------------------------------------------------

// Whether the chunk sums go through FFT correlations (launch_chunk_sums: LT = n -
// M lags a tile), and the transform's size and tiles: the cheaper by a model of
// both, the transforms at 18 TFLOP/s against 8 M flop per lag at k_caf_lags' 64.
// Measured on 20 captures of 65536 samples, 4192 lags and chunks of 512: 732 us
// direct, 73 through the FFTs (the model: 730 and 90).
static bool coarse_fft(const dg_ctx *c, int nmax, int M, int nb_max, int nlag_cap, MapArgs &f)
{
    if (nmax > (1 << 24) || M < 32) return false;  // tiles of a multiple of 32 lags
    double best = (double)((nlag_cap + 895) / 896 * 896) * nb_max * 8.0 * M / 64.0;
    bool fft = false;
    const double budget = (double)(c->opt.scratch_mib ? c->opt.scratch_mib : 12288) * 1048576.0;
    for (int logn = 10; logn <= 14; ++logn) {
        const int n = 1 << logn, lt = n - M;
        if (lt < M) continue;
        const int nt = (nlag_cap + lt - 1) / lt, nwin = nb_max + (nt - 1) * (lt / M);
        const double cost = 5.0 * n * logn * ((double)nb_max + nwin + (double)nb_max * nt) / 18.0;
        if (nt > 65535 || cost >= best || 8.0 * c->K * ((double)nb_max + nwin) * n > budget) continue;
        best = cost;
        fft = true;
        f.logn = logn;
        f.LT = lt;
        f.ntile = nt;
        f.nwin = nwin;
    }
    return fft;
}

dg_status dg_coarse_maps(dg_ctx *c, int32_t bins, int32_t chunk, float *maps)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!maps) return fail(c, DG_EINVAL, "maps is NULL");
    if (c->gd.row0 != 0 || c->gd.nrows != c->gd.nlat)
        return fail(c, DG_EUNSUPPORTED, "dg_coarse_maps needs a context over the whole grid (no row shard)");
    if (c->gd.nlat < 2 || c->gd.nlon < 2) return fail(c, DG_EINVAL, "dg_coarse_maps needs at least 2 x 2 nodes");
    if (bins != 0 && (bins < 2 || bins > 256)) return fail(c, DG_EINVAL, "bins %d outside 2..256 (0: auto)", bins);
    if (chunk != 0 && (chunk < 1 || chunk > 4096 || (chunk & (chunk - 1))))
        return fail(c, DG_EINVAL, "chunk %d is not a power of two in 1..4096 (0: auto)", chunk);
    int nmax = 0;
    for (int k = 0; k < c->K; ++k) {
        if (!c->steps[k].loaded) return fail(c, DG_ESTATE, "snapshot %d has not been loaded", k);
        nmax = std::max(nmax, (int)c->steps[k].n);
    }
    const size_t KG = (size_t)c->K * (size_t)c->G, K = (size_t)c->K;
    CoarseBufs &b = c->co;
    dg_status st = need_nodes(c);
    if (st != DG_OK) return st;
    b.Q = 0;  // the last maps' buffers may go
    if ((st = ensure(c, (void **)&b.lag, &b.lag_cap, sizeof(int) * KG)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.nu, &b.nu_cap, sizeof(float) * KG)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.lmm, &b.lmm_cap, sizeof(int) * 2 * K)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.nmm, &b.nmm_cap, sizeof(unsigned long long) * 2 * K)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.st, &b.st_cap, sizeof(CoarseStep) * K)) != DG_OK) return st;
    if ((st = push_steps(c)) != DG_OK) return st;
    if ((st = ensure_ephf(c)) != DG_OK) return st;
    if ((st = ensure_xyzf(c, c->G)) != DG_OK) return st;
    CoarseArgs a{};
    a.xyz = c->xyz;
    a.xyzf = c->cd.xyzf;
    a.ephf = c->cd.ephf;
    a.fsc_hi = (float)(c->fs / kC);
    a.fsc_lo = (float)(c->fs / kC - (double)a.fsc_hi);
    a.ilf_hi = (float)(1.0 / (c->lambda * c->fs));
    a.ilf_lo = (float)(1.0 / (c->lambda * c->fs) - (double)a.ilf_hi);
    a.G = c->G;
    a.nlat = c->gd.nlat;
    a.nlon = c->gd.nlon;
    a.eph = c->eph;
    a.steps = c->steps_d;
    a.K = c->K;
    a.fs = c->fs;
    a.lambda = c->lambda;
    a.lag = b.lag;
    a.nu = b.nu;
    a.lmm = b.lmm;
    a.nmm = b.nmm;
    a.st = b.st;
    a.maps = maps;
    a.err = c->err_d;
    {  // under way while the host plans (its lattice takes longer on a new grid)
        Timed t(c, DG_K_COARSE);
        int n = 1;
        CK(c, launch_ecef_split(c->xyz, c->G, c->cd.xyzf, c->stream));
        CK(c, launch_coarse_geo(a, c->stream, &n));
        t.done(n);
    }
    // planning from the host's lattice estimate of the FDOA span (25 % margin)
    std::vector<double> &spans = c->cd.main_span;  // cached until the grid changes
    if (spans.size() != K) fdoa_spans(c, c->gd, spans);
    double span = 0.0;
    for (int k = 0; k < c->K; ++k) span = std::max(span, spans[k]);
    span *= 1.25;
    int M = chunk;
    if (M == 0) {  // the chunk's phase error (nu_q - nu_c) m stays below 1/8 cycle
        M = 1024;
        while (M > 1 && 0.5 * span * M > 0.125) M >>= 1;
    }
    int Q = bins;
    if (Q == 0) {  // two bins per Doppler resolution cell 1 / N
        Q = (int)std::ceil(2.0 * nmax * span) + 1;
        Q = std::min(256, std::max(16, (Q + 7) / 8 * 8));
    }
    const int nb_max = (nmax + M - 1) / M;
    if (nb_max > 65535) return fail(c, DG_EUNSUPPORTED, "chunk %d leaves %d chunks (at most 65535)", M, nb_max);
    const double diam = grid_diameter(c->gd);
    int nlag_cap = 0;
    for (int k = 0; k < c->K; ++k) nlag_cap = std::max(nlag_cap, lag_slots(c->eph_host[k], c->fs, diam));
    MapArgs f{};
    bool fft = coarse_fft(c, nmax, M, nb_max, nlag_cap, f);
    a.Q = Q;
    a.M = M;
    a.nlag_cap = nlag_cap;
    a.nb_max = nb_max;
    a.nh_max = (nb_max + 1) / 2;
    a.Dpad = coarse_dpad(Q);
    if ((st = ensure(c, (void **)&b.P, &b.P_cap, sizeof(float2) * K * nb_max * (size_t)nlag_cap)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.A, &b.A_cap, sizeof(float) * K * (size_t)nlag_cap * Q)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.pool, &b.pool_cap, sizeof(float) * K * (size_t)nlag_cap * Q)) != DG_OK) return st;
    if ((st = ensure(c, (void **)&b.turn, &b.turn_cap, sizeof(float4) * K * a.nh_max * (size_t)(a.Dpad / 2))) != DG_OK)
        return st;
    if ((st = ensure(c, (void **)&b.part, &b.part_cap, sizeof(double) * K * coarse_parts(nlag_cap, Q))) != DG_OK)
        return st;
    a.P = b.P;
    a.A = b.A;
    a.pool = b.pool;
    a.turn = b.turn;
    a.part = b.part;
    bool c64 = false;
    for (int k = 0; k < c->K; ++k) c64 |= c->steps[k].fmt == DG_IQ_C64;
    if (fft) {
        const size_t n = (size_t)1 << f.logn;
        st = ensure(c, (void **)&b.snap, &b.snap_cap, sizeof(MapSnap) * K);
        if (st == DG_OK) st = ensure(c, (void **)&b.F2, &b.F2_cap, sizeof(float2) * K * ((size_t)nb_max + f.nwin) * n);
        if (st == DG_OK && c64) st = ensure(c, (void **)&b.bad, &b.bad_cap, sizeof(int) * 4 * K);
        if (st == DG_OK) st = ensure(c, (void **)&b.tw, &b.tw_cap, sizeof(float2) * n, &b.tw_logn);
        if (st != DG_OK && st != DG_ENOMEM) return st;
        if (st == DG_ENOMEM) {  // the direct kernel needs none of these
            c->err.clear();
            fft = false;
        }
    }
    if (fft) {
        if (b.tw_logn != f.logn) {
            b.tw_logn = 0;
            CK(c, launch_map_twiddles(b.tw, f.logn, c->stream));
            ++c->launches;
            b.tw_logn = f.logn;
        }
        a.snap = b.snap;
        a.bad = c64 ? b.bad : nullptr;
        f.sd = c->steps_d;
        f.snap = b.snap;
        f.S = f.ksd = c->K;
        f.Cmax = nb_max;
        f.Mb = M;
        f.NLpad = nlag_cap;
        f.tw = b.tw;
        f.F2 = b.F2;
        f.U = b.P;
        f.bad = c64 ? b.bad : nullptr;
    }
    {
        Timed t(c, DG_K_COARSE);
        int n = 0;
        CK(c, launch_coarse(a, fft ? &f : nullptr, c->stream, &n));
        t.done(n);
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    b.Q = Q;
    b.M = M;
    b.nlag_cap = nlag_cap;
    b.nb_max = nb_max;
    return DG_OK;
}

dg_status dg_coarse_inspect(dg_ctx *c, float *caf, dg_coarse_step *steps, int32_t *shape)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    const CoarseBufs &b = c->co;
    if (b.Q == 0) return fail(c, DG_ESTATE, "no coarse maps have been computed on this context");
    if (shape) {
        shape[0] = b.Q;
        shape[1] = b.M;
        shape[2] = b.nlag_cap;
    }
    if (caf) {
        CK(c, launch_coarse_transpose(b.A, caf, c->K, b.Q, b.nlag_cap, c->stream));
        ++c->launches;
    }
    if (steps) {
        std::vector<CoarseStep> h(c->K);
        CK(c, cudaMemcpyAsync(h.data(), b.st, sizeof(CoarseStep) * c->K, cudaMemcpyDeviceToHost, c->stream));
        CK(c, cudaStreamSynchronize(c->stream));
        for (int k = 0; k < c->K; ++k) {
            steps[k].l0 = h[k].l0;
            steps[k].nlag = h[k].nlag;
            steps[k].nu_lo = h[k].nu_lo;
            steps[k].delta = h[k].delta;
            steps[k].nu_c = h[k].nu_c;
            steps[k].mu = h[k].mu;
        }
        return check_latched(c);
    }
    return DG_OK;
}

// ---------------------------------------------------------------------------
// Search of several regions with one host synchronisation.
// ---------------------------------------------------------------------------

// Bounds of D and the FDOA over a region in every snapshot from 3 x 3 nodes of
// it (field_curvature); false where none hold.
static bool region_range(const dg_ctx *c, const GridDev &g, GridRange *out)
{
    // three columns bound less than half a turn
    if (std::fabs(g.lat0_rad) + 0.5 * g.nlat * g.dlat_m / 6.33e6 > 1.39 || lon_extent(g) > 3.0) return false;
    double p[9][3], hi = 0.0, hj = 0.0;
    auto norm = [](double x, double y, double z) { return std::sqrt(x * x + y * y + z * z); };
    auto dist = [&](int a, int b) { return norm(p[a][0] - p[b][0], p[a][1] - p[b][1], p[a][2] - p[b][2]); };
    for (int q = 0; q < 9; ++q) host_node_ecef(g, 0.5 * (q / 3) * (g.nlat - 1), 0.5 * (q % 3) * (g.nlon - 1), p[q]);
    for (int q = 0; q < 9; ++q) {
        if (q < 6) hi = std::max(hi, dist(q, q + 3));
        if (q % 3 < 2) hj = std::max(hj, dist(q, q + 1));
    }
    const double h = 0.5 * 1.05 * std::hypot(hi, hj) + 1.0;
    const double fc = c->fs / kC, lf = c->lambda * c->fs;
    for (int k = 0; k < c->K; ++k) {
        const dg_ephem &e = c->eph_host[k];
        GridRange R{};
        R.d_lo = R.nu_lo = 1e300;
        R.d_hi = R.nu_hi = -1e300;
        double rmin = 1e300;
        for (int q = 0; q < 9; ++q) {
            double rho[2], uv[2];
            for (int t = 0; t < 2; ++t) {
                const double *pp = t ? e.p2 : e.p1, *vv = t ? e.v2 : e.v1;
                const double x = pp[0] - p[q][0], y = pp[1] - p[q][1], z = pp[2] - p[q][2];
                rho[t] = norm(x, y, z);
                uv[t] = (x * vv[0] + y * vv[1] + z * vv[2]) / rho[t];
            }
            const double D = (rho[1] - rho[0]) * fc, nu = (uv[0] - uv[1]) / lf;
            R.d_lo = std::min(R.d_lo, D);
            R.d_hi = std::max(R.d_hi, D);
            R.nu_lo = std::min(R.nu_lo, nu);
            R.nu_hi = std::max(R.nu_hi, nu);
            rmin = std::min(rmin, std::min(rho[0], rho[1]));
        }
        const double sep = norm(e.p2[0] - e.p1[0], e.p2[1] - e.p1[1], e.p2[2] - e.p1[2]);
        const double dv = norm(e.v2[0] - e.v1[0], e.v2[1] - e.v1[1], e.v2[2] - e.v1[2]);
        const double v = std::max(norm(e.v1[0], e.v1[1], e.v1[2]), norm(e.v2[0], e.v2[1], e.v2[2]));
        const double m = rmin - h - 0.5 * sep;
        if (!(m > 0.0)) return false;
        const Curvature q = field_curvature(c, m, sep, v, dv);
        R.d_lo -= 0.5 * q.d * h * h;
        R.d_hi += 0.5 * q.d * h * h;
        R.nu_lo -= 0.5 * q.nu * h * h;
        R.nu_hi += 0.5 * q.nu * h * h;
        out[k] = R;
    }
    return true;
}

// The surfaces and argmax records of all regions through shared launches:
// table s of the batch is of capture s % K and region s / K. *done = false
// where the maps do not serve these regions.
static dg_status regions_map(dg_ctx *c, const dg_grid *regions, int n, float *costs, bool *done, bool *nodes)
{
    *done = *nodes = false;
    const int64_t G = (int64_t)regions[0].nlat * regions[0].nlon;
    if (!map_options(c) || G < kMapMinNodes || c->gd.row0 != 0 || c->gd.nrows != c->grid.nlat) return DG_OK;
    const size_t K = (size_t)c->K;
    std::vector<GridDev> grids((size_t)n);
    std::vector<GridRange> range(K * (size_t)n);
    for (int r = 0; r < n; ++r) grids[(size_t)r] = make_griddev(regions[r], 0, regions[r].nlat);
    dg_status st;
    // every region's nodes at once, under way while the host plans
    const bool all = n <= 64 && (double)n * G * 24.0 <= 256e6;
    if ((st = ensure(c, (void **)&c->reg_grids, &c->reg_grids_cap, sizeof(GridDev) * (size_t)n)) != DG_OK) return st;
    CK(c, cudaMemcpyAsync(c->reg_grids, grids.data(), sizeof(GridDev) * (size_t)n, cudaMemcpyHostToDevice, c->stream));
    if (all) {
        if ((st = ensure(c, (void **)&c->reg_xyz, &c->reg_xyz_cap, sizeof(double) * 3 * (size_t)G * n)) != DG_OK) return st;
        if ((st = ensure(c, (void **)&c->reg_steps, &c->reg_steps_cap, sizeof(GridStep) * (size_t)n)) != DG_OK) return st;
        Timed t(c, DG_K_GRID);
        CK(c, launch_grid_ecef(grids[0], c->reg_xyz, c->stream, nullptr, c->reg_grids, n, c->reg_steps));
        t.done(1);
    }
    for (int r = 0; r < n; ++r)
        if (!region_range(c, grids[(size_t)r], &range[K * (size_t)r])) return DG_OK;
    MapPlan m;
    std::vector<MapSnap> snap;
    if (!map_shape(c, range, snap, m)) return DG_OK;
    const double budget = (double)(c->opt.scratch_mib ? c->opt.scratch_mib : 12288) * 1048576.0;
    const int nr = (int)std::min((double)std::min(n, (int)(65535 / K)), std::floor(budget / ((double)K * map_bytes(m))));
    if (nr < 1) return DG_OK;
    // the tables of the main grid's plan are replaced, also where the search fails
    // later on: the plan, and graphs and batches that replay on them, are stale
    c->mp.gen = 0;
    ++c->steps_gen;
    if ((st = map_buffers(c, m, K * (size_t)nr, snap)) != DG_OK) return st;
    if ((st = push_steps(c)) != DG_OK) return st;
    if (!all) {
        if ((st = ensure(c, (void **)&c->reg_xyz, &c->reg_xyz_cap, sizeof(double) * 3 * (size_t)G * nr)) != DG_OK) return st;
        if ((st = ensure(c, (void **)&c->reg_steps, &c->reg_steps_cap, sizeof(GridStep) * (size_t)nr)) != DG_OK) return st;
    }
    if ((st = ensure(c, &c->amax_tmp, &c->amax_tmp_bytes, argmax_tmp_bytes(G) * (size_t)nr)) != DG_OK) return st;
    for (int r0 = 0; r0 < n; r0 += nr) {
        const int R = std::min(nr, n - r0);
        const double *xyz = c->reg_xyz + (all ? 3 * G * r0 : 0);
        const GridStep *steps = c->reg_steps + (all ? r0 : 0);
        if (!all) {
            Timed t(c, DG_K_GRID);
            CK(c, launch_grid_ecef(grids[0], c->reg_xyz, c->stream, nullptr, c->reg_grids + r0, R, c->reg_steps));
            t.done(1);
        }
        MapArgs a{};
        map_common(c, 0, xyz, grids[0], G, a);
        map_tables_args(m, c->mb, a);
        a.ksd = c->K;
        a.nreg = R;
        a.S = c->K * R;
        a.snap = c->mb.snap + K * (size_t)r0;
        a.first = 1;
        a.out = costs + G * r0;
        {
            Timed t(c, DG_K_CDFT_CONTRACT);
            int nl = 1;
            CK(c, launch_map_tables(a, c->stream, &nl));
            CK(c, launch_map_expand(a, c->stream));
            t.done(nl);
        }
        {
            Timed t(c, DG_K_CDFT_COMBINE);
            CK(c, launch_map_lookup(a, c->stream));
            t.done(1);
        }
        {
            Timed t(c, DG_K_ARGMAX);
            int nl = 0;
            CK(c, launch_argmax(a.out, G, DG_PREC_FP32, grids[0], steps, c->amax_tmp, c->reg_res + r0, &nl, c->stream,
                                nullptr, c->reg_grids + r0, R));
            t.done(nl);
        }
    }
    CK(c, cudaMemcpyAsync(c->err_h, c->err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    c->last_map = true;
    c->cd_chunk_min = c->cd_chunk_max = -1;
    c->mp.rows = 0;
    for (size_t k = 0; k < K; ++k) c->mp.rows += (int64_t)snap[k].NL * ((c->steps[k].n + m.Mb - 1) / m.Mb);
    *done = true;
    *nodes = all;
    return DG_OK;
}

// The refinement around the best of n regions, whose records are on the device, up
// to its fix in fix_host_sync, with nothing read by the host in between. *done =
// false (and nothing kept) where refine_map does not serve it.
static dg_status refine_best(dg_ctx *c, const dg_grid *regions, int n, double spacing_m, int half, bool *done)
{
    *done = false;
    if (half == 0 || !map_options(c)) return DG_OK;
    std::vector<GridDev> mains((size_t)n);
    for (int r = 0; r < n; ++r) mains[(size_t)r] = make_griddev(regions[r], 0, regions[r].nlat);
    dg_status st = ensure_post(c, half, &c->fix_dev_sync, &c->fix_host_sync);
    if (st != DG_OK) return st;
    const int side = 2 * half + 1;
    dg_grid lg = regions[0];  // the centre is replaced on the device
    lg.dlat_m = lg.dlon_m = spacing_m;
    lg.nlat = lg.nlon = side;
    const GridDev lgd = make_griddev(lg, 0, side);
    const int64_t Gl = (int64_t)side * side;
    {
        Timed t(c, DG_K_REFINE);
        CK(c, launch_best_record(c->reg_res, n, c->amax_res, c->stream));
        CK(c, launch_grid_ecef(lgd, c->loc.xyz, c->stream, c->amax_res, nullptr, 1, c->gstep + 1));
        t.done(2);
    }
    if ((st = refine_map(c, lgd, c->loc.xyz, Gl, c->loc.cost, done, mains.data(), n)) != DG_OK || !*done) return st;
    {
        Timed t(c, DG_K_ARGMAX);
        int nl = 0;
        CK(c, launch_argmax(c->loc.cost, Gl, c->opt.prec, lgd, c->gstep + 1, c->amax_tmp, c->amax_fine, &nl, c->stream,
                            c->amax_res, nullptr, 1, FixOut{c->fix_dev_sync, c->amax_res, mains[0], side}));
        t.done(nl);
    }
    CK(c, cudaMemcpyAsync(c->fix_host_sync, c->fix_dev_sync, sizeof(dg_fix), cudaMemcpyDeviceToHost, c->stream));
    return DG_OK;
}

dg_status dg_search_regions(dg_ctx *c, const dg_grid *regions, int32_t n, void *costs, double spacing_m,
                            double window_m, dg_fix *out, int32_t *best)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!regions || !costs || !out) return fail(c, DG_EINVAL, "regions, costs and out must not be NULL");
    if (n < 1 || n > 256) return fail(c, DG_EINVAL, "n = %d outside 1..256", n);
    for (int r = 0; r < n; ++r) {
        dg_status st = validate_grid(c, &regions[r]);
        if (st != DG_OK) return st;
        if (regions[r].nlat != regions[0].nlat || regions[r].nlon != regions[0].nlon)
            return fail(c, DG_EINVAL, "regions must all have the same number of nodes");
    }
    for (int k = 0; k < c->K; ++k)
        if (!c->steps[k].loaded) return fail(c, DG_ESTATE, "snapshot %d has not been loaded", k);
    const int64_t G = (int64_t)regions[0].nlat * regions[0].nlon;
    const size_t esz = c->opt.prec == DG_PREC_FP64 ? 8 : 4;
    if (c->reg_cap < (size_t)n) {
        c->reg_cap = 0;
        c->reg_n = 0;
        if (c->reg_res) CK(c, cudaFreeAsync(c->reg_res, c->stream));
        c->reg_res = nullptr;
        if (c->reg_host) {
            CK(c, cudaStreamSynchronize(c->stream));
            cudaFreeHost(c->reg_host);
            c->reg_host = nullptr;
        }
        CK(c, device_alloc(c, &c->reg_res, sizeof(ArgmaxResult) * n));
        CK(c, pinned_alloc(&c->reg_host, sizeof(ArgmaxResult) * n));
        c->reg_cap = (size_t)n;
    }
    dg_status st;
    bool done = false, nodes = false;
    c->reg_n = 0;
    st = regions_map(c, regions, n, (float *)costs, &done, &nodes);
    if (st == DG_ENOMEM) {  // no memory for all regions' tables: one region after the other
        c->err.clear();
        done = nodes = false;
    } else if (st != DG_OK) {
        return st;
    }
    for (int r = 0; r < n && !done; ++r) {
        if ((st = dg_set_grid(c, &regions[r])) != DG_OK) return st;
        if ((st = ensure_surf(c)) != DG_OK) return st;
        if ((st = ensure(c, &c->amax_tmp, &c->amax_tmp_bytes, argmax_tmp_bytes(G))) != DG_OK) return st;
        void *cr = (char *)costs + esz * (size_t)G * r;
        if ((st = run_surface(c, c->gd, c->xyz, G, c->surf, cr, false)) != DG_OK) return st;
        int nl = 0;
        {
            Timed t(c, DG_K_ARGMAX);
            CK(c, launch_argmax(cr, G, c->opt.prec, c->gd, c->gstep, c->amax_tmp, c->reg_res + r, &nl, c->stream));
            t.done(nl);
        }
    }
    CK(c, cudaMemcpyAsync(c->reg_host, c->reg_res, sizeof(ArgmaxResult) * n, cudaMemcpyDeviceToHost, c->stream));
    int half = 0;
    bool refined = false;
    if (done && refine_half(c, spacing_m, window_m, &half) == DG_OK &&
        (st = refine_best(c, regions, n, spacing_m, half, &refined)) != DG_OK)
        return st;
    CK(c, cudaStreamSynchronize(c->stream));
    if ((st = check_latched(c)) != DG_OK) return st;
    c->reg_n = n;
    int b = -1;
    for (int r = 0; r < n; ++r)
        if (c->reg_host[r].idx >= 0 && (b < 0 || c->reg_host[r].val > c->reg_host[b].val)) b = r;
    if (b < 0) return fail(c, DG_EINVAL, "no region holds a finite value");
    // the best region becomes the context's grid; its nodes are there already
    if ((st = set_grid(c, &regions[b], nodes ? c->reg_xyz + 3 * G * b : nullptr, nodes ? c->reg_steps + b : nullptr)) != DG_OK)
        return st;
    if (refined) {
        if ((st = copy_fix(c, c->fix_host_sync, out)) != DG_OK) return st;
        if (best) *best = b;
        return DG_OK;
    }
    if ((st = argmax_refine(c, (char *)costs + esz * (size_t)G * b, spacing_m, window_m, out, c->reg_res + b)) != DG_OK)
        return st;
    if (best) *best = b;
    return DG_OK;
}

dg_status dg_region_maxima(dg_ctx *c, double *out, int32_t n)
{
    if (!c) return fail(nullptr, DG_EINVAL, "ctx is NULL");
    c->err.clear();
    if (!out) return fail(c, DG_EINVAL, "out is NULL");
    if (n < 1 || n > c->reg_n) return fail(c, DG_ESTATE, "the last search had %d regions, not %d", c->reg_n, n);
    for (int r = 0; r < n; ++r) out[r] = c->reg_host[r].idx >= 0 ? c->reg_host[r].val : std::nan("");
    return DG_OK;
}

}  // extern "C"

extern "C" dg_status dg_debug_tc_wait_limit(uint32_t polls)
{
    g_tc_wait_polls.store(polls, std::memory_order_relaxed);
    return DG_OK;
}
