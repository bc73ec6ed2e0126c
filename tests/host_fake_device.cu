// The library's host code (csrc/dg_api.cu) over a fake device: allocations are
// host memory that can be made to fail, and every launch checks, in place of its
// kernels, that the buffers it was given are alive, large enough and hold what
// the kernels read. Run by test_host_allocations.py; no GPU is used.
#include "dg_api.cu"

#include <cstdlib>
#include <functional>

namespace fake {
std::map<char *, size_t> blocks;
long allocations = 0, fail_at = 0, fail_count = 1;  // fail allocations fail_at .. fail_at + fail_count - 1
bool failed = false, capturing = false;
int sorts = 0;      // lag sorts launched
bool busy = false;  // a batch's replay still runs
cudaError_t error = cudaSuccess;  // what cudaGetLastError returns, once

cudaError_t last()
{
    const cudaError_t e = error;
    error = cudaSuccess;
    return e;
}
std::string op;
int faults = 0;

void fault(const char *what, const char *which)
{
    if (++faults <= 20) std::printf("FAULT in %s: %s %s (allocation %ld fails)\n", op.c_str(), what, which, fail_at);
}
cudaError_t alloc(void **p, size_t bytes)
{
    if (capturing) fault("allocation", "under capture");
    ++allocations;
    if (fail_at && allocations >= fail_at && allocations < fail_at + fail_count) {
        failed = true;  // *p stays as it is
        return error = cudaErrorMemoryAllocation;
    }
    char *q = (char *)std::malloc(bytes ? bytes : 1);
    std::memset(q, 0xa5, std::min(bytes, (size_t)1 << 16));
    blocks[q] = bytes;
    *p = q;
    return cudaSuccess;
}
cudaError_t release(void *p)
{
    if (!p) return cudaSuccess;
    if (!blocks.erase((char *)p)) {
        fault("free of", "a buffer that is not alive");
        return cudaErrorInvalidValue;
    }
    std::free(p);
    return cudaSuccess;
}
bool holds(const void *p, double bytes)
{
    auto it = blocks.upper_bound((char *)p);
    if (it == blocks.begin()) return false;
    --it;
    return (char *)p + (size_t)bytes <= it->first + it->second;
}
bool need(const void *p, double bytes, const char *name)
{
    if (bytes <= 0 || holds(p, bytes)) return true;
    fault("buffer", name);
    return false;
}
}  // namespace fake

#define NEED(p, n) fake::need(p, sizeof(*(p)) * (double)(n), #p)
#define SAME(x, y, name) \
    if (!(std::fabs((double)(x) - (double)(y)) < 1e-3)) fake::fault("contents of", name)

// a definition of a runtime function under its link name only (its headers hold a
// device version of some that a second definition would collide with)
#define RUNTIME(ret, name, args)             \
    ret fake_##name args __asm__("" #name); \
    ret fake_##name args

extern "C" {
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
RUNTIME(cudaError_t, cudaMallocAsync, (void **p, size_t n, cudaStream_t)) { return fake::alloc(p, n); }
RUNTIME(cudaError_t, cudaMalloc, (void **p, size_t n)) { return fake::alloc(p, n); }
RUNTIME(cudaError_t, cudaMallocHost, (void **p, size_t n)) { return fake::alloc(p, n); }
RUNTIME(cudaError_t, cudaFreeAsync, (void *p, cudaStream_t)) { return fake::release(p); }
RUNTIME(cudaError_t, cudaFree, (void *p)) { return fake::release(p); }
RUNTIME(cudaError_t, cudaFreeHost, (void *p)) { return fake::release(p); }
RUNTIME(cudaError_t, cudaMemcpyAsync, (void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t))
{
    // a pinned host buffer is one of the blocks, a pageable one is not
    if (kind == cudaMemcpyDeviceToHost && (size_t)d < 4096) fake::fault("buffer", "copy's destination");
    if ((size_t)d < 4096 || (size_t)s < 4096) return cudaSuccess;
    if (kind != cudaMemcpyDeviceToHost && !fake::need(d, (double)n, "copy's destination")) return cudaSuccess;
    if (kind != cudaMemcpyHostToDevice && !fake::need(s, (double)n, "copy's source")) return cudaSuccess;
    std::memmove(d, s, n);
    return cudaSuccess;
}
RUNTIME(cudaError_t, cudaMemcpy, (void *d, const void *s, size_t n, cudaMemcpyKind k)) { return fake_cudaMemcpyAsync(d, s, n, k, 0); }
RUNTIME(cudaError_t, cudaMemsetAsync, (void *d, int v, size_t n, cudaStream_t))
{
    if (fake::need(d, (double)n, "memset")) std::memset(d, v, n);
    return cudaSuccess;
}
RUNTIME(cudaError_t, cudaStreamSynchronize, (cudaStream_t))
{
    if (fake::capturing) fake::fault("synchronisation", "under capture");
    return cudaSuccess;
}
RUNTIME(cudaError_t, cudaGetDevice, (int *d)) { return *d = 0, cudaSuccess; }
RUNTIME(cudaError_t, cudaDeviceGetAttribute, (int *v, cudaDeviceAttr, int)) { return *v = 152, cudaSuccess; }
RUNTIME(cudaError_t, cudaGetLastError, ()) { return fake::last(); }
RUNTIME(const char *, cudaGetErrorString, (cudaError_t)) { return "fake error"; }
RUNTIME(cudaError_t, cudaEventCreate, (cudaEvent_t *e)) { return *e = (cudaEvent_t)1, cudaSuccess; }
RUNTIME(cudaError_t, cudaEventCreateWithFlags, (cudaEvent_t *e, unsigned)) { return *e = (cudaEvent_t)1, cudaSuccess; }
RUNTIME(cudaError_t, cudaEventDestroy, (cudaEvent_t)) { return cudaSuccess; }
RUNTIME(cudaError_t, cudaEventElapsedTime, (float *t, cudaEvent_t, cudaEvent_t)) { return *t = 1.f, cudaSuccess; }
RUNTIME(cudaError_t, cudaEventRecord, (cudaEvent_t, cudaStream_t)) { return cudaSuccess; }
RUNTIME(cudaError_t, cudaEventSynchronize, (cudaEvent_t)) { return cudaSuccess; }
RUNTIME(cudaError_t, cudaEventQuery, (cudaEvent_t))
{
    return fake::busy ? fake::error = cudaErrorNotReady : cudaSuccess;
}
RUNTIME(cudaError_t, cudaStreamWaitEvent, (cudaStream_t, cudaEvent_t, unsigned)) { return cudaSuccess; }
RUNTIME(cudaError_t, cudaStreamBeginCapture, (cudaStream_t, cudaStreamCaptureMode)) { return fake::capturing = true, cudaSuccess; }
RUNTIME(cudaError_t, cudaStreamEndCapture, (cudaStream_t, cudaGraph_t *g))
{
    fake::capturing = false;
    return *g = (cudaGraph_t)1, cudaSuccess;
}
RUNTIME(cudaError_t, cudaGraphInstantiate, (cudaGraphExec_t *e, cudaGraph_t, unsigned long long))
{
    return *e = (cudaGraphExec_t)1, cudaSuccess;
}
RUNTIME(cudaError_t, cudaGraphDestroy, (cudaGraph_t)) { return cudaSuccess; }
RUNTIME(cudaError_t, cudaGraphExecDestroy, (cudaGraphExec_t)) { return cudaSuccess; }
RUNTIME(cudaError_t, cudaGraphLaunch, (cudaGraphExec_t, cudaStream_t)) { return cudaSuccess; }
}

namespace dg {
static void captures(const StepDesc *sd, int S)
{
    if (!NEED(sd, S)) return;  // and what they point to
    for (int s = 0; s < S; ++s) {
        fake::need(sd[s].y1, (double)iq_bytes(sd[s].fmt) * sd[s].n, "y1");
        fake::need(sd[s].y2, (double)iq_bytes(sd[s].fmt) * sd[s].n, "y2");
    }
}
static void geometry_inputs(const double *xyz, const double *eph, const float *ephf, int S, double nodes)
{
    NEED(xyz, 3 * nodes);
    if (NEED(eph, 12 * S) && ephf && NEED(ephf, 24 * S))
        for (int i = 0; i < 12 * S; ++i) SAME((double)ephf[2 * i] + ephf[2 * i + 1] - eph[i], 0.0, "ephf");
}
static void bases(const CdftBatch &a)
{
    if (!NEED(a.bbase, a.S + 1) || !NEED(a.gbase, a.S + 1)) return;
    for (int s = 0; s < a.S; ++s)
        if (a.bbase[s + 1] <= a.bbase[s] || a.gbase[s + 1] <= a.gbase[s]) fake::fault("contents of", "lag slots");
}
cudaError_t launch_cdft_geo(const CdftBatch &a, cudaStream_t)
{
    const double SG = (double)a.S * a.G;
    geometry_inputs(a.xyz, a.eph, a.ephf, a.S, (double)a.G);
    NEED(a.xyzf, 6 * a.G);
    NEED(a.lr, 2 * a.S), NEED(a.nur, 2 * a.S), NEED(a.candL, SG), NEED(a.candNu, SG), NEED(a.err, 1);
    if (a.delay != DG_DELAY_INTEGER) NEED(a.candMu, SG);
    return fake::last();
}
cudaError_t launch_ecef_split(const double *xyz, int64_t G, float *xyzf, cudaStream_t, int *lr, unsigned *nur, int S)
{
    NEED(xyz, 3 * G), NEED(xyzf, 6 * G);
    if (lr) NEED(lr, 2 * S), NEED(nur, 2 * S);
    return fake::last();
}
static void sorted(const CdftBatch &a)
{
    ++fake::sorts;
    const double SG = (double)a.S * a.G;
    bases(a);
    NEED(a.candL, SG), NEED(a.candNu, SG), NEED(a.order, SG), NEED(a.nuS, SG), NEED(a.g2b, a.ngroups);
    if (a.delay != DG_DELAY_INTEGER) NEED(a.muS, SG);
}
cudaError_t launch_sort_small(const CdftBatch &a, cudaStream_t) { return sorted(a), fake::last(); }
cudaError_t launch_cdft_plan(const CdftBatch &a, int NBT, cudaStream_t)
{
    sorted(a);
    NEED(a.count, NBT), NEED(a.offs, NBT), NEED(a.subcnt, NBT), NEED(a.need, NBT);
    NEED(a.nubase, a.S), NEED(a.delta, a.S);
    if (!a.mma) NEED(a.V, (double)a.S * a.M * 64);
    return fake::last();
}
cudaError_t launch_corr_lag(const CdftBatch &a, int nseg, int, float *surf, float2 *part, cudaStream_t)
{
    captures(a.sd, a.S);
    sorted(a);
    if (part) NEED(part, (double)a.S * nseg * a.G);
    else NEED(surf, (double)(a.k0 + a.S) * a.G);
    return fake::last();
}
cudaError_t launch_corr_segments(const float2 *part, int S, int nseg, int64_t G, int, float *surf, float *out, cudaStream_t)
{
    NEED(part, (double)S * nseg * G);
    if (out) NEED(out, G);
    else NEED(surf, (double)S * G);
    return fake::last();
}
cudaError_t launch_corr_direct(const CorrArgs &a, cudaStream_t)
{
    captures(a.steps, a.K);
    geometry_inputs(a.xyz, a.eph, nullptr, a.K, (double)a.G);
    fake::need(a.surf, (a.prec == DG_PREC_FP64 ? 8.0 : 4.0) * a.K * a.G, "surf");
    return fake::last();
}
cudaError_t launch_accumulate(const void *surf, int K, int64_t G, int prec, void *out, cudaStream_t)
{
    const double e = prec == DG_PREC_FP64 ? 8.0 : 4.0;
    fake::need(surf, e * K * G, "surf"), fake::need(out, e * G, "out");
    return fake::last();
}
cudaError_t launch_cdft_tiles(const CdftBatch &a, cudaStream_t)
{
    bases(a);
    NEED(a.tbase, a.S + 1), NEED(a.hbase, a.S + 1), NEED(a.layout, a.S), NEED(a.Mcs, a.S);
    return fake::last();
}
static cudaError_t contract(const CdftBatch &a, int fmt)
{
    for (int s = 0; NEED(a.sd, a.S) && s < a.S; ++s)
        if (a.sd[s].fmt != fmt) fake::fault("a capture", "of another format than its batch's");
    captures(a.sd, a.S);
    bases(a);
    NEED(a.tbase, a.S + 1), NEED(a.nubase, a.S), NEED(a.delta, a.S);
    if (NEED(a.bbase, a.S + 1)) NEED(a.W, (double)a.bbase[a.S] * a.Bmax * 128), NEED(a.need, a.bbase[a.S]);
    return fake::last();
}
cudaError_t launch_cdft_contract_fp32(const CdftBatch &a, int, int fmt, cudaStream_t) { return contract(a, fmt); }
cudaError_t launch_cdft_contract_mma(const CdftBatch &a, int, int fmt, int, cudaStream_t) { return contract(a, fmt); }
cudaError_t launch_cdft_contract_hankel(const CdftBatch &a, int, int fmt, int, cudaStream_t) { return contract(a, fmt); }
size_t cdft_btab_bytes(int, int M) { return (size_t)M * 256; }
cudaError_t launch_cdft_btab(const CdftBatch &a, int mode, void *btab, cudaStream_t)
{
    fake::need(btab, (double)a.S * cdft_btab_bytes(mode, a.M), "btab");
    return fake::last();
}
cudaError_t launch_cdft_superchunk(const CdftBatch &a, int NBT, cudaStream_t)
{
    NEED(a.W, (double)NBT * a.Bmax * 128);
    return fake::last();
}
cudaError_t launch_cdft_combine(const CdftBatch &a, float *surf, cudaStream_t)
{
    sorted(a);
    NEED(surf, (double)(a.k0 + a.S) * a.G);
    return fake::last();
}
TcJob tc_job(const CdftBatch &a, const void *btab)
{
    TcJob j{};
    j.W = a.W;
    j.btab = btab;
    return j;
}
cudaError_t launch_tc_job_tiles(const TcJob *j, int n, int *t, cudaStream_t) { return NEED(j, n), NEED(t, n + 1), fake::last(); }
cudaError_t launch_cdft_contract_jobs(const TcJob *j, int n, const int *t, int, int, int, unsigned, cudaStream_t)
{
    NEED(j, n), NEED(t, n + 1);
    return fake::last();
}

// the twiddles carry their length, the node polynomials and the fit are partitions of unity
cudaError_t launch_map_twiddles(float2 *tw, int logn, cudaStream_t)
{
    if (NEED(tw, 1 << logn)) tw[0] = make_float2((float)logn, 0.f);
    return fake::last();
}
static void twiddles(const MapArgs &a)
{
    if (NEED(a.tw, 1 << a.logn)) SAME(a.tw[0].x, a.logn, "tw");
}
static void tables(const MapArgs &a)
{
    const double S = a.S;
    captures(a.sd, a.ksd);
    twiddles(a);
    if (NEED(a.T, a.P * a.Q))
        for (int q = 0; q < a.Q; ++q) {
            double sum = 0.0;
            for (int p = 0; p < a.P; ++p) sum += a.T[p * a.Q + q];
            SAME(sum, 1.0, "T");
        }
    if (NEED(a.snap, a.S))
        for (int s = 0; s < a.S; ++s)
            if (a.snap[s].NL < 1 || a.snap[s].NL > a.NLpad || a.snap[s].NL > a.ntile * a.LT) fake::fault("contents of", "snap");
    NEED(a.F2, S * a.ntile * a.Cmax * (1 << a.logn)), NEED(a.U, S * a.Cmax * a.P * a.NLpad);
    NEED(a.X, S * a.Q * a.NLpad), NEED(a.phase, S * a.Cmax * a.Q);
    if (a.bad) NEED(a.bad, 4 * a.ksd);
}
cudaError_t launch_map_tables(const MapArgs &a, cudaStream_t, int *n) { return tables(a), *n += 2, fake::last(); }
cudaError_t launch_map_expand(const MapArgs &a, cudaStream_t) { return tables(a), fake::last(); }
cudaError_t launch_map_poly(const MapArgs &a, cudaStream_t)
{
    geometry_inputs(a.xyz, a.eph, a.ephf, a.ksd, (double)a.G);
    if (NEED(a.fit, kPolyTerms * kPolyPts))
        for (int t = 0; t < kPolyTerms; ++t) {
            double sum = 0.0;
            for (int i = 0; i < kPolyPts; ++i) sum += a.fit[t * kPolyPts + i];
            SAME(sum, t == 0 ? 1.0 : 0.0, "fit");
        }
    const double tiles = std::ceil((double)a.nrows / a.poly.rows) * std::ceil((double)a.nlon / kPolyCols);
    NEED(a.coef, tiles * a.S * kPolyStride);
    return fake::last();
}
cudaError_t launch_map_lookup(const MapArgs &a, cudaStream_t)
{
    geometry_inputs(a.xyz, a.eph, a.ephf, a.ksd, (double)a.G * a.nreg);
    NEED(a.X, (double)a.S * a.Q * a.NLpad), NEED(a.out, (double)a.G * a.nreg), NEED(a.snap, a.S);
    return fake::last();
}
size_t map_few_partials(int P, int NL) { return (size_t)((NL + 3) / 4) * 8 * P; }
cudaError_t launch_map_few(const MapArgs &a, const MapFew &f, cudaStream_t, int *n)
{
    captures(a.sd, a.S);
    NEED((float *)a.U, map_few_partials(a.P, a.LT) * (double)a.Cmax * a.S);
    NEED(f.snap, a.S), NEED(a.X, (double)a.S * a.Q * a.NLpad);
    *n += 2;
    return fake::last();
}
cudaError_t launch_detect(const void *v, int, const GridDev &g, const GridStep *step, double, int, int cap, int max_peaks,
                          int *count, int64_t *cand, DetectPeak *out, cudaStream_t)
{
    fake::need(v, 4.0 * g.nrows * g.nlon, "cost");
    if (NEED(step, 1) && NEED(count, 1) && NEED(cand, cap) && NEED(out, max_peaks)) *count = 0;
    return fake::last();
}
size_t argmax_tmp_bytes(int64_t n) { return (size_t)(n + 1023) / 1024 * 16; }
cudaError_t launch_argmax(const void *v, int64_t n, int, const GridDev &, const GridStep *step, void *tmp, ArgmaxResult *res,
                          int *launches, cudaStream_t, const ArgmaxResult *centre, const GridDev *grids, int ngrids, FixOut fin)
{
    fake::need(v, 4.0 * n * ngrids, "cost"), fake::need(tmp, (double)argmax_tmp_bytes(n) * ngrids, "argmax_tmp");
    NEED(step, ngrids);
    if (grids) NEED(grids, ngrids);
    if (centre) NEED(centre, 1);
    if (NEED(res, ngrids))
        for (int r = 0; r < ngrids; ++r) res[r] = ArgmaxResult{1.0, 0, 0.8, 0.1, 0.8, 0.1};
    if (fin.fix && NEED(fin.fix, 1)) std::memset(fin.fix, 0, sizeof *fin.fix);
    *launches += 1;
    return fake::last();
}
cudaError_t launch_best_record(const ArgmaxResult *r, int n, ArgmaxResult *out, cudaStream_t)
{
    if (NEED(r, n) && NEED(out, 1)) *out = r[0];
    return fake::last();
}
cudaError_t launch_grid_ecef(const GridDev &g, double *xyz, cudaStream_t, const ArgmaxResult *centre, const GridDev *grids,
                             int ngrids, GridStep *step_out)
{
    NEED(xyz, 3.0 * g.nrows * g.nlon * ngrids);
    if (centre) NEED(centre, 1);
    if (grids) NEED(grids, ngrids);
    if (step_out) NEED(step_out, ngrids);
    return fake::last();
}
cudaError_t launch_step_geometry(const GridDev &g, const double *xyz, const double *eph, double, double, int, int *, double *,
                                 double *, cudaStream_t)
{
    geometry_inputs(xyz, eph, nullptr, 1, (double)g.nrows * g.nlon);
    return fake::last();
}
int coarse_parts(int cap, int) { return (cap + 31) / 32; }
int coarse_dpad(int Q) { return (Q + 31) / 32 * 32; }
cudaError_t launch_coarse_geo(const CoarseArgs &a, cudaStream_t, int *)
{
    const double KG = (double)a.K * a.G;
    geometry_inputs(a.xyz, a.eph, a.ephf, a.K, (double)a.G);
    NEED(a.xyzf, 6 * a.G), NEED(a.lag, KG), NEED(a.nu, KG), NEED(a.lmm, 2 * a.K), NEED(a.nmm, 2 * a.K);
    return fake::last();
}
cudaError_t launch_coarse(const CoarseArgs &a, const MapArgs *f, cudaStream_t, int *)
{
    const double m = (double)a.K * a.nlag_cap;
    captures(a.steps, a.K);
    NEED(a.P, m * a.nb_max), NEED(a.A, m * a.Q), NEED(a.pool, m * a.Q), NEED(a.st, a.K);
    NEED(a.turn, (double)a.K * a.nh_max * a.Dpad / 2), NEED(a.part, (double)a.K * coarse_parts(a.nlag_cap, a.Q));
    NEED(a.maps, (double)a.K * (a.nlat - 1) * (a.nlon - 1));
    if (f) {
        twiddles(*f);
        NEED(f->snap, a.K), NEED(f->F2, (double)a.K * (f->Cmax + f->nwin) * (1 << f->logn)), NEED(f->U, m * f->Cmax);
        if (f->bad) NEED(f->bad, 4 * a.K);
    }
    return fake::last();
}
cudaError_t launch_coarse_transpose(const float *A, float *out, int K, int Q, int cap, cudaStream_t)
{
    NEED(A, (double)K * Q * cap), NEED(out, (double)K * Q * cap);
    return fake::last();
}
}  // namespace dg

// ---------------------------------------------------------------------------
static dg_grid grid_of(int n, int m, double spacing)
{
    dg_grid g{};
    g.lat0_deg = 45.0;
    g.lon0_deg = 10.0;
    g.dlat_m = g.dlon_m = spacing;
    g.nlat = n;
    g.nlon = m;
    return g;
}

// The calls of a program that goes through several grids, lengths and windows, one
// after the other whatever each returns; true if every one returned DG_OK.
static bool program(const dg_options &o, const std::vector<dg_grid> &grids, int K)
{
    std::vector<dg_ephem> eph((size_t)K);
    for (int k = 0; k < K; ++k) {  // 550 km above the grid, moving east
        const double r = 6.92e6, la = 45.0 * kPi / 180.0, lo = (10.0 + 0.05 * k) * kPi / 180.0;
        for (int t = 0; t < 2; ++t) {
            const double l = lo + 0.008 * t, v = 7500.0;
            double *p = t ? eph[k].p2 : eph[k].p1, *w = t ? eph[k].v2 : eph[k].v1;
            p[0] = r * std::cos(la) * std::cos(l), p[1] = r * std::cos(la) * std::sin(l), p[2] = r * std::sin(la);
            w[0] = -v * std::sin(l), w[1] = v * std::cos(l), w[2] = 300.0;
        }
    }
    bool good = true;
    dg_ctx *c = nullptr;
    auto call = [&](const char *name, dg_status st) {
        if (st != DG_OK && st != DG_ENOMEM) {
            const char *e = dg_last_error(c);
            fake::fault(e ? e : "", name);
        }
        good = good && st == DG_OK;
    };
    fake::op = "dg_create";
    dg_status st = dg_create(&grids[0], eph.data(), K, 12.5e6, 1575.42e6, &o, (void *)0x100, &c);
    call("dg_create", st);
    if (st != DG_OK) return false;
    const int nmax = 20000;
    std::vector<float> y((size_t)2 * nmax, 1.f);
    const size_t cells = 1 << 18;  // of each of up to eight snapshots
    float *cost = (float *)std::malloc(sizeof(float) * 8 * cells), *maps = (float *)std::malloc(sizeof(float) * 8 * cells);
    fake::blocks[(char *)cost] = sizeof(float) * 8 * cells;
    fake::blocks[(char *)maps] = sizeof(float) * 8 * cells;
    dg_fix fix;
    dg_peak peaks[4];
    int32_t np = 0, best = 0;
    auto load = [&](int n) {
        fake::op = "dg_load_capture";
        for (int k = 0; k < K; ++k)
            for (int tries = 0; tries < 8; ++tries) {
                const dg_status s = dg_load_capture(c, k, DG_IQ_C64, y.data(), y.data(), n, 0);
                call("dg_load_capture", s);
                if (s == DG_OK) break;
            }
    };
    load(3000);
    for (const dg_grid &g : grids)
        for (const dg_grid *h : {&g, &grids[0]}) {  // back to a shape that the context knows
            fake::op = "dg_set_grid";
            call("dg_set_grid", dg_set_grid(c, h));
            fake::op = "dg_cost_surface";
            call("dg_cost_surface", dg_cost_surface(c, cost));
            fake::op = "dg_coarse_maps";
            call("dg_coarse_maps", dg_coarse_maps(c, 0, 0, maps));
        }
    for (int n : {3000, nmax})
        for (const dg_grid &g : grids) {
            load(n);
            fake::op = "dg_set_grid";
            call("dg_set_grid", dg_set_grid(c, &g));
            fake::op = "dg_cost_surface";
            call("dg_cost_surface", dg_cost_surface(c, cost));
            for (double window : {100.0, 1000.0}) {
                fake::op = "dg_argmax_refine";
                call("dg_argmax_refine", dg_argmax_refine(c, cost, 20.0, window, &fix));
            }
            fake::op = "dg_detect";
            call("dg_detect", dg_detect(c, cost, 0.5, 1, 2, 4, peaks, &np));
            fake::op = "dg_coarse_maps";
            call("dg_coarse_maps", dg_coarse_maps(c, 0, 0, maps));
            fake::op = "dg_graph_capture";
            st = dg_graph_capture(c, cost, 20.0, 200.0);
            call("dg_graph_capture", st);
            if (st == DG_OK) {
                fake::op = "dg_graph_launch";
                call("dg_graph_launch", dg_graph_launch(c));
                call("dg_graph_fix", dg_graph_fix(c, &fix));
            }
            for (int side : {95, 21}) {
                std::vector<dg_grid> r(3, grid_of(side, side, 0.4 * g.dlat_m));
                for (int i = 0; i < 3; ++i) r[(size_t)i].lat0_deg += 0.2 * i;
                fake::op = "dg_search_regions";
                call("dg_search_regions", dg_search_regions(c, r.data(), 3, cost, 20.0, 200.0, &fix, &best));
            }
            fake::op = "dg_set_grid";
            call("dg_set_grid", dg_set_grid(c, &g));
            fake::op = "dg_cost_surface (again)";
            call("dg_cost_surface", dg_cost_surface(c, cost));
        }
    // what failed before works now
    if (fake::failed) {
        fake::fail_at = 0;
        for (const dg_grid &g : grids) {
            fake::op = "after the failure";
            if (dg_set_grid(c, &g) != DG_OK || dg_cost_surface(c, cost) != DG_OK || dg_coarse_maps(c, 0, 0, maps) != DG_OK ||
                dg_argmax_refine(c, cost, 20.0, 200.0, &fix) != DG_OK || dg_graph_capture(c, cost, 20.0, 200.0) != DG_OK)
                fake::fault(dg_last_error(c), "after the failure");
        }
    }
    fake::op = "dg_destroy";
    dg_destroy(c);
    fake::blocks.erase((char *)cost);
    fake::blocks.erase((char *)maps);
    std::free(cost);
    std::free(maps);
    return good;
}

// The grouped direct surface keeps its sort within the scratch target, and a surface
// that finds no memory for it is computed on the tiles.
static void direct_scratch()
{
    dg_options o;
    dg_options_default(&o);
    const dg_grid g = grid_of(300, 301, 200.0);
    const double G = 300.0 * 301.0;
    const int K = 3, n = 4096;
    std::vector<dg_ephem> eph((size_t)K);
    for (dg_ephem &e : eph) {
        e = dg_ephem{};
        e.p1[0] = e.p2[0] = 6.9e6;
        e.p2[1] = 5e4;
        e.v1[1] = e.v2[1] = 7500.0;
    }
    std::vector<float> y((size_t)2 * n, 1.f);
    float *cost = (float *)std::malloc(4 * (size_t)G);
    fake::blocks[(char *)cost] = 4 * (size_t)G;
    auto live = [] {
        double b = 0.0;
        for (const auto &x : fake::blocks) b += (double)x.second;
        return b;
    };
    struct {
        int mib, fail;
        bool sorted;
    } cases[] = {{0, 0, true}, {1, 0, false}, {4, 0, false}, {9, 0, true}, {16, 0, true}, {0, 2, false}, {0, 5, false}};
    for (const auto &t : cases) {
        fake::op = "direct scratch " + std::to_string(t.mib) + " " + std::to_string(t.fail);
        o.scratch_mib = t.mib;
        dg_ctx *c = nullptr;
        if (dg_create(&g, eph.data(), K, 12.5e6, 1575.42e6, &o, (void *)0x100, &c) != DG_OK) fake::fault("dg_create", "");
        for (int k = 0; k < K; ++k) dg_load_capture(c, k, DG_IQ_C64, y.data(), y.data(), n, 0);
        const double before = live() + 4.0 * K * G;
        fake::allocations = 0;
        fake::fail_at = t.fail;
        fake::sorts = 0;
        for (int r = 0; r < 2; ++r, fake::fail_at = 0)
            if (dg_cost_surface(c, cost) != DG_OK) fake::fault("dg_cost_surface", dg_last_error(c));
        const double used = live() - before;
        if ((fake::sorts > 0) != t.sorted) fake::fault("the wrong kernel", "");
        if (t.mib && used > 1048576.0 * t.mib + 65536.0) fake::fault("scratch beyond its target", std::to_string(used).c_str());
        dg_destroy(c);
    }
    fake::blocks.erase((char *)cost);
    std::free(cost);
}

// Buffers replaced while a captured step may read them are kept, and given back once
// it cannot be launched and does not run any more: a program that alternates between
// windows and grids beside its graph or batch holds no more and more of them.
static void kept_buffers(bool cdft)
{
    dg_options o;
    dg_options_default(&o);
    if (cdft) {
        o.algo = DG_ALGO_CDFT;
        o.contract = DG_CONTRACT_FP16X3;
        o.chunk = 512;
    }
    const dg_grid a = grid_of(40, 41, 200.0), b = grid_of(44, 45, 300.0);
    const int K = 2, n = 4096;
    std::vector<dg_ephem> eph((size_t)K);
    for (dg_ephem &e : eph) {
        e = dg_ephem{};
        e.p1[0] = e.p2[0] = 6.9e6;
        e.p2[1] = 5e4;
        e.v1[1] = e.v2[1] = 7500.0;
    }
    std::vector<float> y((size_t)2 * n, 1.f);
    float *cost = (float *)std::malloc(4 * 45 * 45);
    fake::blocks[(char *)cost] = 4 * 45 * 45;
    dg_ctx *c = nullptr;
    dg_fix fix;
    fake::fail_at = 0;
    auto ok = [&](dg_status st, const char *what) {
        if (st != DG_OK) fake::fault(dg_last_error(c), what);
    };
    ok(dg_create(&a, eph.data(), K, 12.5e6, 1575.42e6, &o, (void *)0x100, &c), "dg_create");
    for (int k = 0; k < K; ++k) ok(dg_load_capture(c, k, DG_IQ_C64, y.data(), y.data(), n, 0), "dg_load_capture");
    auto windows = [&](int times) {
        for (int i = 0; i < times; ++i)
            for (double w : {60.0, 100.0, 140.0}) {
                ok(dg_cost_surface(c, cost), "dg_cost_surface");
                ok(dg_argmax_refine(c, cost, 20.0, w, &fix), "dg_argmax_refine");
            }
    };
    auto grids = [&](int times) {
        for (int i = 0; i < times; ++i)
            for (const dg_grid *g : {&b, &a}) {
                ok(dg_set_grid(c, g), "dg_set_grid");
                windows(1);
            }
    };
    auto growth = [&](const char *what, auto f) {  // blocks that 20 further rounds add
        fake::op = what;
        f(2);
        const size_t before = fake::blocks.size();
        f(20);
        if (fake::blocks.size() > before) fake::fault(what, "keeps more and more buffers");
        return fake::blocks.size();
    };
    const size_t none = growth("no captured step", grids);
    fake::op = "another format";  // the batches of snapshots have one each
    for (int k : {1, 0, 1}) {
        ok(dg_load_capture(c, k, k ? DG_IQ_CI8 : DG_IQ_C64, y.data(), y.data(), n, 0), "dg_load_capture");
        windows(1);
    }
    ok(dg_load_capture(c, 1, DG_IQ_C64, y.data(), y.data(), n, 0), "dg_load_capture");
    windows(1);
    ok(dg_graph_capture(c, cost, 20.0, 60.0), "dg_graph_capture");
    growth("windows beside a graph", windows);
    ok(dg_graph_launch(c), "dg_graph_launch");
    if (growth("grids beside a stale graph", grids) > none + 2) fake::fault("a stale graph", "keeps its buffers");
    dg_batch *bt = nullptr;
    void *costs[1] = {cost};
    ok(dg_batch_capture(&c, 1, costs, 20.0, 60.0, (void *)0x200, &bt), "dg_batch_capture");
    growth("windows beside a batch", windows);
    ok(dg_batch_launch(bt), "dg_batch_launch");
    fake::busy = true;  // its replay still reads the old grid's tables
    const size_t at = fake::blocks.size();
    grids(1);
    if (fake::blocks.size() <= at) fake::fault("a running batch", "lost its buffers");
    fake::busy = false;
    if (growth("grids beside a stale batch", grids) > none + 2) fake::fault("a stale batch", "keeps its buffers");
    dg_batch_destroy(bt);
    dg_destroy(c);
    fake::blocks.erase((char *)cost);
    std::free(cost);
    fake::op = "the end";
    if (!fake::blocks.empty()) fake::fault("buffers never given back,", std::to_string(fake::blocks.size()).c_str());
}

int main(int argc, char **argv)
{
    if (argc > 1 && std::string(argv[1]).rfind("kept", 0) == 0) {
        kept_buffers(std::string(argv[1]) == "kept-cdft");
        return fake::faults ? 1 : 0;
    }
    if (argc > 1 && std::string(argv[1]) == "scratch") {
        direct_scratch();
        return fake::faults ? 1 : 0;
    }
    dg_options o;
    dg_options_default(&o);
    const std::string what = argc > 1 ? argv[1] : "maps";
    const int count = argc > 2 ? std::atoi(argv[2]) : 1;
    // grids of other lags, bins and geometry, down and up in size
    std::vector<dg_grid> grids = {grid_of(93, 95, 150.0), grid_of(95, 99, 3000.0), grid_of(40, 40, 800.0)};
    if (what == "maps") grids.push_back(grid_of(322, 1000, 20.0));  // polynomial geometry
    if (what != "direct") {
        o.algo = DG_ALGO_CDFT;
        o.contract = what == "fp32" ? DG_CONTRACT_FP32 : DG_CONTRACT_FP16X3;
        if (what == "chunks") o.chunk = 512;
        if (what == "lagrange") o.delay = DG_DELAY_LAGRANGE4;
    }
    long runs = 0;
    fake::fail_count = count;
    fake::fail_at = 0;
    if (!program(o, grids, 3)) fake::fault("an error", "without a failed allocation");
    for (long f = 1;; ++f, ++runs) {
        fake::allocations = 0;
        fake::failed = false;
        fake::error = cudaSuccess;
        fake::fail_at = f;
        program(o, grids, 3);
        if (!fake::failed) break;
    }
    fake::op = "the end";
    fake::fail_at = 0;
    if (!fake::blocks.empty()) fake::fault("buffers never given back,", std::to_string(fake::blocks.size()).c_str());
    std::printf("%s: %ld runs with failed allocations, %d faults\n", what.c_str(), runs, fake::faults);
    return fake::faults ? 1 : 0;
}
