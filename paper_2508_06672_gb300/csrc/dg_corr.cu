// dg_corr.cu -- direct position-domain correlation (Sec. III, Eq. 11).
//
// One CTA handles one tile of candidates (kWarps*R grid rows x 32 grid
// columns) for one snapshot k; R, the candidates (grid rows) per thread, is a
// launch choice (dg_options.rows, tuned by dg_autotune). FP32 with integer delays runs
// here only where few candidates share a lag, captures are longer than 2^24 samples or
// the sort finds no room (run_surface_lag); k_corr_lag below takes the rest. Per
// candidate it computes the geometry (Eq. 3-10, FP64), then
//     C = sum_n y1[n] conj(y2~[n]) exp(j 2 pi nu n),
// y2~[n] = y2[n + L] (Eq. 9) or its 4-tap Lagrange interpolation at n + D,
// and writes |C|^2 (or |C|) into the snapshot's slice of the per-snapshot
// surface buffer; a separate pass sums the snapshots in order.
//
// Sum evaluation: y1 is staged in shared memory already multiplied by
// (-j)^n, which moves the wanted frequency to theta = 2 pi nu + pi/2. The
// sum over n of x[n] exp(j theta n) is then run as a second-order resonator
//     s[n] = x[n] + 2 cos(theta) s[n-1] - s[n-2],
//     sum  = exp(j theta (n_end-1)) (s[n_end-1] - exp(j theta) s[n_end-2]),
// with x[n] = y1'[n] conj(y2~[n]) folded into the same FMAs: 6 FMAs per
// candidate and sample, no per-sample phasor. Near theta = pi/2 the
// resonator is well conditioned (|nu| <= 0.2 is enforced). The closing phase
// is reduced in FP64.
//
// Shared memory holds a chunk of y1 (M samples) and the window of y2 that
// every candidate of the tile needs for that chunk (M + lag span + taps),
// converted to float/double; the captures stay L2-resident across CTAs.
#include <climits>

#include "dg_internal.cuh"

namespace dg {

template <typename T> struct Cx;
template <> struct Cx<float> { using t = float2; };
template <> struct Cx<double> { using t = double2; };

// M-sample chunks of y1 and a W-sample y2 window in shared memory.
template <typename T> struct Cfg;
template <> struct Cfg<float> { static constexpr int M = 2048, W = 4096; };
template <> struct Cfg<double> { static constexpr int M = 1024, W = 2048; };

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

template <typename C2> __device__ __forceinline__ C2 mk(double x, double y);
template <> __device__ __forceinline__ float2 mk<float2>(double x, double y) { return make_float2((float)x, (float)y); }
template <> __device__ __forceinline__ double2 mk<double2>(double x, double y) { return make_double2(x, y); }

template <typename T, int FMT>
__device__ __forceinline__ typename Cx<T>::t load_c(const void *b, int idx)
{
    const float2 v = IQ<FMT>::load(b, idx);
    return mk<typename Cx<T>::t>(v.x, v.y);
}

// Resonator update for two consecutive samples: (a0, b0) then (a1, b1).
// On entry s1 = s[n-1], s2 = s[n-2]; on exit s1 = s[n+1], s2 = s[n].
template <typename T, typename C2>
__device__ __forceinline__ void resonate2(const C2 &a0, const C2 &b0, const C2 &a1, const C2 &b1,
                                          T c2, C2 &s1, C2 &s2)
{
    // x = a * conj(b) = (a.x b.x + a.y b.y, a.y b.x - a.x b.y)
    s2.x = fma_(c2, s1.x, fma_(a0.y, b0.y, fma_(a0.x, b0.x, -s2.x)));
    s2.y = fma_(c2, s1.y, fma_(-a0.x, b0.y, fma_(a0.y, b0.x, -s2.y)));
    s1.x = fma_(c2, s2.x, fma_(a1.y, b1.y, fma_(a1.x, b1.x, -s1.x)));
    s1.y = fma_(c2, s2.y, fma_(-a1.x, b1.y, fma_(a1.y, b1.x, -s1.y)));
}

template <typename T, typename C2>
__device__ __forceinline__ C2 interp4(const C2 *q, const T *w)
{
    C2 r;
    r.x = fma_(w[3], q[3].x, fma_(w[2], q[2].x, fma_(w[1], q[1].x, w[0] * q[0].x)));
    r.y = fma_(w[3], q[3].y, fma_(w[2], q[2].y, fma_(w[1], q[1].y, w[0] * q[0].y)));
    return r;
}

// y2~ at sample n for lag L read straight from global memory (fallback when
// the tile's lag span does not fit the shared-memory window).
template <typename T, int FMT, int DELAY>
__device__ __forceinline__ typename Cx<T>::t y2_global(const void *y2, int N, int n, int L, const T *w)
{
    using C2 = typename Cx<T>::t;
    if constexpr (DELAY == DG_DELAY_INTEGER) {
        const int q = n + L;
        return (q >= 0 && q < N) ? load_c<T, FMT>(y2, q) : mk<C2>(0.0, 0.0);
    } else {
        C2 t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = n + L - 1 + u;
            t[u] = (q >= 0 && q < N) ? load_c<T, FMT>(y2, q) : mk<C2>(0.0, 0.0);
        }
        return interp4<T, C2>(t, w);
    }
}

template <typename T, int FMT, int DELAY, int R>
__global__ void __launch_bounds__(kThreads) k_corr_direct(CorrArgs a, int tiles_j)
{
    using C2 = typename Cx<T>::t;
    constexpr int MCH = Cfg<T>::M, WIN = Cfg<T>::W;
    constexpr int TAPS = (DELAY == DG_DELAY_LAGRANGE4) ? 3 : 0;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *y1s = reinterpret_cast<C2 *>(smem_raw);
    C2 *y2s = y1s + MCH;
    __shared__ int s_min[kWarps], s_max[kWarps];

    const int k = blockIdx.y;
    const int ti = blockIdx.x / tiles_j, tj = blockIdx.x % tiles_j;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // For each r the 32 lanes of a warp take a compact 4-row x 8-column patch
    // (warp w: columns 8 (w % 4) .. + 7 of the tile, rows 4R (w / 4) .. + 4R - 1;
    // lane: column lane % 8, row lane / 8, then 4 rows further per r). Their
    // lags then differ by at most 10 grid steps' worth, not 31 as along one
    // row, so the y2 window reads of a warp stay within a few banks' rows
    // where a grid step moves the lag by a sample or more.
    static_assert(kWarps == 8, "the lane mapping assumes 8 warps: 4 column blocks x 2 row blocks");
    const int j = tj * 32 + (warp & 3) * 8 + (lane & 7);
    const int row0 = ti * (kWarps * R) + (warp >> 2) * (4 * R) + (lane >> 3);
    const StepDesc sd = a.steps[k];
    const int N = sd.n;
    const int64_t G = a.G;

    double e[12];
#pragma unroll
    for (int t = 0; t < 12; ++t) e[t] = __ldg(a.eph + 12 * k + t);

    // ---- geometry of this thread's R candidates (FP64) ---------------------
    int off[R];
    T c2[R];
    T w[R][4];
    bool ok[R];
    int lmin = INT_MAX, lmax = INT_MIN;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = row0 + 4 * r;
        ok[r] = (i < a.nrows) && (j < a.nlon);
        off[r] = 0;
        c2[r] = (T)0;
        w[r][0] = (T)0; w[r][1] = (T)1; w[r][2] = (T)0; w[r][3] = (T)0;
        if (ok[r]) {
            const int64_t p = (int64_t)i * a.nlon + j;
            double D, nu;
            geometry(a.xyz[p], a.xyz[G + p], a.xyz[2 * G + p], e, a.fs, a.lambda, D, nu);
            if (!(fabs(nu) <= 0.2)) {
                atomicOr(a.err, ERR_NU_RANGE);
                ok[r] = false;
            } else if (!(fabs(D) < 1.0e9)) {
                atomicOr(a.err, ERR_LAG_RANGE);
                ok[r] = false;
            } else {
                const int L = lag_of(D, DELAY);
                off[r] = L;
                c2[r] = (T)(-2.0 * sinpi(2.0 * nu));
                if (DELAY == DG_DELAY_LAGRANGE4) {
                    const double mu = D - (double)L;
                    w[r][0] = (T)(-mu * (mu - 1.0) * (mu - 2.0) / 6.0);
                    w[r][1] = (T)((mu + 1.0) * (mu - 1.0) * (mu - 2.0) / 2.0);
                    w[r][2] = (T)(-(mu + 1.0) * mu * (mu - 2.0) / 2.0);
                    w[r][3] = (T)((mu + 1.0) * mu * (mu - 1.0) / 6.0);
                }
                lmin = min(lmin, L);
                lmax = max(lmax, L);
            }
        }
    }
    // ---- tile lag range --------------------------------------------------------
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        lmin = min(lmin, __shfl_xor_sync(0xffffffffu, lmin, d));
        lmax = max(lmax, __shfl_xor_sync(0xffffffffu, lmax, d));
    }
    if (lane == 0) {
        s_min[warp] = lmin;
        s_max[warp] = lmax;
    }
    __syncthreads();
    lmin = s_min[0];
    lmax = s_max[0];
#pragma unroll
    for (int u = 1; u < kWarps; ++u) {
        lmin = min(lmin, s_min[u]);
        lmax = max(lmax, s_max[u]);
    }
    if (lmin > lmax) return;  // no valid candidate in the tile (uniform)
    const int span = lmax - lmin;
    int mch = MCH;
    if (span + TAPS + MCH > WIN) mch = ((WIN - span - TAPS) / 64) * 64;
    const bool windowed = mch >= 64;
    if (!windowed) mch = MCH;
#pragma unroll
    for (int r = 0; r < R; ++r) off[r] = ok[r] ? off[r] - lmin : 0;

    C2 s1[R], s2[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        s1[r] = mk<C2>(0.0, 0.0);
        s2[r] = mk<C2>(0.0, 0.0);
    }

    // ---- sample loop -----------------------------------------------------------
    for (int n0 = 0; n0 < N; n0 += mch) {
        const int len = min(mch, N - n0);
        const int len2 = (len + 1) & ~1;
        __syncthreads();
        for (int q = threadIdx.x; q < len2; q += kThreads) {
            const int n = n0 + q;
            C2 v = (n < N) ? load_c<T, FMT>(sd.y1, n) : mk<C2>(0.0, 0.0);
            C2 o;
            switch (n & 3) {  // multiply by (-j)^n
            case 0: o = v; break;
            case 1: o.x = v.y; o.y = -v.x; break;
            case 2: o.x = -v.x; o.y = -v.y; break;
            default: o.x = -v.y; o.y = v.x; break;
            }
            y1s[q] = o;
        }
        if (windowed) {
            const int base = n0 + lmin - (TAPS ? 1 : 0);
            const int wl = len2 + span + TAPS;
            for (int q = threadIdx.x; q < wl; q += kThreads) {
                const int n = base + q;
                y2s[q] = (n >= 0 && n < N) ? load_c<T, FMT>(sd.y2, n) : mk<C2>(0.0, 0.0);
            }
        }
        __syncthreads();
        if (windowed) {
            if (DELAY == DG_DELAY_INTEGER) {
#pragma unroll 4
                for (int m = 0; m < len2; m += 2) {
                    const C2 a0 = y1s[m], a1 = y1s[m + 1];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const C2 *q = y2s + m + off[r];
                        resonate2<T, C2>(a0, q[0], a1, q[1], c2[r], s1[r], s2[r]);
                    }
                }
            } else {
#pragma unroll 2
                for (int m = 0; m < len2; m += 2) {
                    const C2 a0 = y1s[m], a1 = y1s[m + 1];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const C2 *q = y2s + m + off[r];
                        const C2 b0 = interp4<T, C2>(q, w[r]);
                        const C2 b1 = interp4<T, C2>(q + 1, w[r]);
                        resonate2<T, C2>(a0, b0, a1, b1, c2[r], s1[r], s2[r]);
                    }
                }
            }
        } else {
            for (int m = 0; m < len2; m += 2) {
                const C2 a0 = y1s[m], a1 = y1s[m + 1];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int L = off[r] + lmin;
                    const C2 b0 = y2_global<T, FMT, DELAY>(sd.y2, N, n0 + m, L, w[r]);
                    const C2 b1 = y2_global<T, FMT, DELAY>(sd.y2, N, n0 + m + 1, L, w[r]);
                    resonate2<T, C2>(a0, b0, a1, b1, c2[r], s1[r], s2[r]);
                }
            }
        }
    }

    // ---- close the resonators and write |C|^2 or |C| ---------------------------
    const int nend = (N + 1) & ~1;  // resonator steps taken (zero-padded to even)
    T *surf = reinterpret_cast<T *>(a.surf) + (int64_t)k * G;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (!ok[r]) continue;
        const int i = row0 + 4 * r;
        const int64_t p = (int64_t)i * a.nlon + j;
        double D, nu;
        geometry(a.xyz[p], a.xyz[G + p], a.xyz[2 * G + p], e, a.fs, a.lambda, D, nu);
        // E = exp(j theta (nend-1)) = exp(j 2 pi nu (nend-1)) * j^(nend-1)
        const double ph = nu * (double)(nend - 1);
        double se, ce;
        sincospi(2.0 * (ph - floor(ph)), &se, &ce);
        double ex, ey;
        switch ((nend - 1) & 3) {
        case 0: ex = ce; ey = se; break;
        case 1: ex = -se; ey = ce; break;
        case 2: ex = -ce; ey = -se; break;
        default: ex = se; ey = -ce; break;
        }
        // exp(j theta) = j exp(j 2 pi nu)
        double st, ct;
        sincospi(2.0 * nu, &st, &ct);
        const double thx = -st, thy = ct;
        const double ax = (double)s2[r].x, ay = (double)s2[r].y;
        const double ux = (double)s1[r].x - (thx * ax - thy * ay);
        const double uy = (double)s1[r].y - (thx * ay + thy * ax);
        const double cx = ex * ux - ey * uy;
        const double cy = ex * uy + ey * ux;
        const double pw = cx * cx + cy * cy;
        surf[p] = (T)((a.acc == DG_ACC_POWER) ? pw : sqrt(pw));
    }
}

// ---------------------------------------------------------------------------
// The same sum with the candidates grouped by lag (FP32, integer delay): all
// candidates of a lag share z[n] = y1[n] conj(y2[n + L]), so a warp forms z
// once (32 samples per instruction, into its slice of shared memory) and runs
// the resonators of up to 32 candidates of that lag on broadcast reads of it:
//     s[n] = (z[n] (-j)^n - s[n-2]) + 2 cos(theta) s[n-1];
// with v[n] = s[n] times the signs +, +, -, - the subtraction is an addition,
//     v[n] = (z[n] {1, -j}[n % 2] + v[n-2]) -/+ 2 cos(theta) v[n-1]  (n even / odd):
// one packed addition and one packed FMA per candidate and sample where
// the kernel above issues 6 FMAs and an 8-byte shared load of its own (2
// cycles of the shared-memory port per warp, its bound). The FP32 pipe bounds
// it: 4 operations per candidate-sample (301 x 403 nodes, 4 snapshots of 32768:
// 5.15 -> 2.39 ms). A group costs the same however few candidates it has; where
// that is more than the tiles cost, the kernel above runs (tiles_faster in
// dg_api.cu, both sides measured).
// The lag sort (k_cdft_geo, hist, scan, scatter) gives the groups. Small
// problems split the samples into segments (blockIdx.y) to fill the chip; a
// segment's sum carries its absolute phase and k_corr_segments adds them in
// order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 add_x2(float2 a, float2 b)
{
    unsigned long long r, x, y;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(r));
    return d;
}
__device__ __forceinline__ float2 fma_x2(float2 a, float2 b, float2 c)
{
    unsigned long long r, x, y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(r));
    return d;
}

constexpr int kLagChunk = 128;  // samples of z per warp and pass

// One group's segment by one warp, R candidates per lane.
template <int FMT, int R>
__device__ __forceinline__ void corr_lag_group(const CdftBatch &a, const int4 &gr, const StepDesc &sd, int L, int n0,
                                               int end, float2 *z, float *surf, float2 *part)
{
    const int lane = threadIdx.x & 31, s = gr.y, N = sd.n;
    int cand[R];
    float nu[R];
    float2 cp[R], cn[R], v1[R], v2[R];  // +-2 cos(theta), v[n - 1], v[n - 2]
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const size_t at = (size_t)s * a.G + gr.z + min(lane + 32 * r, gr.w - 1);
        cand[r] = a.order[at];
        nu[r] = a.nuS[at];
        const float c2 = -2.f * sinpif(2.f * nu[r]);
        cp[r] = make_float2(c2, c2);
        cn[r] = make_float2(-c2, -c2);
        v1[r] = v2[r] = make_float2(0.f, 0.f);
    }
    // this lane's samples of the next pass: n0 + lane + 32 i, times -j where n
    // (and so the lane) is odd
    constexpr int E = kLagChunk / 32;
    float2 x[E], y[E];
    auto fetch = [&](int n) {
        if (n + kLagChunk <= end && n + L >= 0 && n + L + kLagChunk <= N) {
#pragma unroll
            for (int i = 0; i < E; ++i) {
                x[i] = IQ<FMT>::load(sd.y1, n + lane + 32 * i);
                y[i] = IQ<FMT>::load(sd.y2, n + lane + 32 * i + L);
            }
        } else {
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const int q = n + lane + 32 * i, r = q + L;
                x[i] = q < end ? IQ<FMT>::load(sd.y1, q) : make_float2(0.f, 0.f);
                y[i] = q < end && r >= 0 && r < N ? IQ<FMT>::load(sd.y2, r) : make_float2(0.f, 0.f);
            }
        }
    };
    fetch(n0);
    for (int n = n0; n < end; n += kLagChunk) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const float zx = fmaf(x[i].x, y[i].x, x[i].y * y[i].y), zy = fmaf(x[i].y, y[i].x, -x[i].x * y[i].y);
            z[lane + 32 * i] = lane & 1 ? make_float2(zy, -zx) : make_float2(zx, zy);
        }
        __syncwarp();
        if (n + kLagChunk < end) fetch(n + kLagChunk);
        const int len = min(kLagChunk, (end - n + 1) & ~1);  // zeros beyond the capture
        const float4 *z4 = reinterpret_cast<const float4 *>(z);
#pragma unroll 8
        for (int m = 0; m < len / 2; ++m) {
            const float4 q = z4[m];
#pragma unroll
            for (int r = 0; r < R; ++r) v2[r] = fma_x2(cn[r], v1[r], add_x2(make_float2(q.x, q.y), v2[r]));
#pragma unroll
            for (int r = 0; r < R; ++r) v1[r] = fma_x2(cp[r], v2[r], add_x2(make_float2(q.z, q.w), v1[r]));
        }
    }
    // the last pair's common sign: + for an even number of pairs before it
    const float sg = (((end - n0 + 1) >> 1) - 1) & 1 ? -1.f : 1.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (lane + 32 * r >= gr.w) continue;
        // close: e^{j theta (n_end - 1)} (s[n_end - 1] - e^{j theta} s[n_end - 2]), e^{j theta} = j e^{j 2 pi nu}
        float st, ct;
        sincospif(2.f * nu[r], &st, &ct);
        const float2 s1 = make_float2(sg * v1[r].x, sg * v1[r].y), s2 = make_float2(sg * v2[r].x, sg * v2[r].y);
        const float ux = s1.x + fmaf(st, s2.x, ct * s2.y), uy = s1.y + fmaf(st, s2.y, -ct * s2.x);
        if (!part) {
            const float pw = fmaf(ux, ux, uy * uy);
            surf[(size_t)(a.k0 + s) * a.G + cand[r]] = a.acc == DG_ACC_POWER ? pw : sqrtf(pw);
        } else {
            const int e = n0 + ((end - n0 + 1) & ~1) - 1;
            float se, ce;
            sincospif(2.f * (frac_mul(nu[r], (float)e) + 0.25f * (float)(e & 3)), &se, &ce);
            part[((size_t)s * gridDim.y + blockIdx.y) * a.G + cand[r]] =
                make_float2(fmaf(ce, ux, -se * uy), fmaf(ce, uy, se * ux));
        }
    }
}

template <int FMT>
__device__ __forceinline__ void corr_lag_fmt(const CdftBatch &a, const int4 &gr, const StepDesc &sd, int L, int n0,
                                             int end, float2 *z, float *surf, float2 *part)
{
    if (gr.w > 32) corr_lag_group<FMT, 2>(a, gr, sd, L, n0, end, z, surf, part);
    else corr_lag_group<FMT, 1>(a, gr, sd, L, n0, end, z, surf, part);
}

__global__ void __launch_bounds__(256) k_corr_lag(CdftBatch a, int seg_len, float *surf, float2 *part)
{
    __shared__ __align__(16) float2 s_z[8][kLagChunk];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t g = blockIdx.x * (int64_t)8 + warp;
    if (g >= a.ngroups) return;
    const int4 gr = a.g2b[g];
    if (gr.x < 0) return;
    const int s = gr.y;
    const StepDesc sd = a.sd[s];
    const int n0 = blockIdx.y * seg_len, N = sd.n;
    if (n0 >= N) {  // a capture shorter than the longest: an empty segment
        for (int i = lane; part && i < gr.w; i += 32)
            part[((size_t)s * gridDim.y + blockIdx.y) * a.G + a.order[(size_t)s * a.G + gr.z + i]] = make_float2(0.f, 0.f);
        return;
    }
    const int end = min(N, n0 + seg_len), L = a.lr[2 * s] + (gr.x - a.bbase[s]);
    if (sd.fmt == DG_IQ_CI16) corr_lag_fmt<DG_IQ_CI16>(a, gr, sd, L, n0, end, s_z[warp], surf, part);
    else if (sd.fmt == DG_IQ_CI8) corr_lag_fmt<DG_IQ_CI8>(a, gr, sd, L, n0, end, s_z[warp], surf, part);
    else corr_lag_fmt<DG_IQ_C64>(a, gr, sd, L, n0, end, s_z[warp], surf, part);
}

// Segment sums to surface values: of each snapshot (surf), or summed over the
// snapshots in order (out).
__global__ void __launch_bounds__(256) k_corr_segments(const float2 *__restrict__ part, int S, int nseg, int64_t G,
                                                       int acc, float *__restrict__ surf, float *__restrict__ out)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < G; p += (int64_t)gridDim.x * blockDim.x) {
        float sum = 0.f;
        for (int s = out ? 0 : blockIdx.y; s < (out ? S : blockIdx.y + 1); ++s) {
            const float2 *q = part + (size_t)s * nseg * G + p;
            float2 c = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int i = 0; i < nseg; ++i) {
                const float2 v = __ldg(q + (size_t)i * G);
                c.x += v.x;
                c.y += v.y;
            }
            float pw = fmaf(c.x, c.x, c.y * c.y);
            if (acc != DG_ACC_POWER) pw = sqrtf(pw);
            if (out) sum = s ? sum + pw : pw;
            else surf[(size_t)s * G + p] = pw;
        }
        if (out) out[p] = sum;
    }
}

cudaError_t launch_corr_lag(const CdftBatch &a, int nseg, int seg_len, float *surf, float2 *part, cudaStream_t s)
{
    k_corr_lag<<<dim3((unsigned)((a.ngroups + 7) / 8), (unsigned)nseg), 256, 0, s>>>(a, seg_len, surf, part);
    return cudaGetLastError();
}

cudaError_t launch_corr_segments(const float2 *part, int S, int nseg, int64_t G, int acc, float *surf, float *out,
                                 cudaStream_t s)
{
    int64_t b = (G + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    k_corr_segments<<<dim3((unsigned)b, out ? 1u : (unsigned)S), 256, 0, s>>>(part, S, nseg, G, acc, surf, out);
    return cudaGetLastError();
}

template <typename T, int FMT, int DELAY, int R>
static cudaError_t launch_one(const CorrArgs &a, cudaStream_t s)
{
    using C2 = typename Cx<T>::t;
    const size_t smem = (size_t)(Cfg<T>::M + Cfg<T>::W) * sizeof(C2);
    // The attribute is per function and device; setting it each launch keeps
    // this correct for every device and thread at negligible cost.
    cudaError_t e = cudaFuncSetAttribute(k_corr_direct<T, FMT, DELAY, R>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int tiles_i = (a.nrows + kWarps * R - 1) / (kWarps * R);
    const int tiles_j = (a.nlon + 31) / 32;
    const int64_t tiles = (int64_t)tiles_i * tiles_j;
    if (tiles > INT_MAX || a.K > 65535) return cudaErrorInvalidValue;
    dim3 grid((unsigned)tiles, (unsigned)a.K);
    k_corr_direct<T, FMT, DELAY, R><<<grid, kThreads, smem, s>>>(a, tiles_j);
    return cudaGetLastError();
}

// Grid rows per thread: FP32 4, 8 or 16; FP64 2 or 4. The defaults are the
// fastest measured on a 1001^2 grid (K = 50, N = 131072): FP32 8 with the
// integer delay (4 and 16 within 1 %), 4 with LAGRANGE4 (5 % ahead of 8).
template <typename T, int FMT, int DELAY>
static cudaError_t launch_rows(const CorrArgs &a, cudaStream_t s)
{
    if constexpr (sizeof(T) == 4) {
        const int rows = a.rows ? a.rows : (DELAY == DG_DELAY_INTEGER ? 8 : 4);
        switch (rows) {
        case 4: return launch_one<T, FMT, DELAY, 4>(a, s);
        case 8: return launch_one<T, FMT, DELAY, 8>(a, s);
        case 16: return launch_one<T, FMT, DELAY, 16>(a, s);
        default: return cudaErrorInvalidValue;
        }
    } else {
        switch (a.rows) {
        case 2: return launch_one<T, FMT, DELAY, 2>(a, s);
        case 0:
        case 4: return launch_one<T, FMT, DELAY, 4>(a, s);
        default: return cudaErrorInvalidValue;
        }
    }
}

template <typename T, int FMT>
static cudaError_t launch_delay(const CorrArgs &a, cudaStream_t s)
{
    return a.delay == DG_DELAY_INTEGER ? launch_rows<T, FMT, DG_DELAY_INTEGER>(a, s)
                                       : launch_rows<T, FMT, DG_DELAY_LAGRANGE4>(a, s);
}

template <typename T>
static cudaError_t launch_fmt(const CorrArgs &a, cudaStream_t s)
{
    switch (a.fmt) {
    case DG_IQ_C64: return launch_delay<T, DG_IQ_C64>(a, s);
    case DG_IQ_CI16: return launch_delay<T, DG_IQ_CI16>(a, s);
    case DG_IQ_CI8: return launch_delay<T, DG_IQ_CI8>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_corr_direct(const CorrArgs &a, cudaStream_t s)
{
    return a.prec == DG_PREC_FP64 ? launch_fmt<double>(a, s) : launch_fmt<float>(a, s);
}

}  // namespace dg
