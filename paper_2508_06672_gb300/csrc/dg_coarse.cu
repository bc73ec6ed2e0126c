// dg_coarse.cu -- coarse delay-Doppler maps of each snapshot, back-projected
// onto the cells of the grid: the input of the learned proposal.
//
// Per snapshot k (captures y1, y2 of n samples; zero outside [0, n)):
//   X(l, nu) = sum_n y1[n] conj(y2[n + l]) e^{j 2 pi nu n}     (Eq. 11 at an
//   integer lag l and FDOA nu: the cross-ambiguity function of the two-step
//   TDOA/FDOA method, Sec. I), sampled at the lags l0 .. l0 + nlag - 1 that
//   the grid's nodes take (Eq. 9) and at Q bins nu_q = nu_lo + q delta over
//   the nodes' FDOA range [nu_lo, nu_hi] (Eq. 10).
// It is evaluated in chunks of M samples turned at the centre frequency
// nu_c = (nu_lo + nu_hi) / 2,
//   P_b(l) = sum_{m<M} y1[bM+m] e^{j 2 pi nu_c (bM+m)} conj(y2[bM+m+l]),
//   Xc(l, q) = sum_b e^{j 2 pi (nu_q - nu_c) b M} P_b(l),
// which is X(l, nu_q) with each sample's phase off by (nu_q - nu_c) m at most
// (M is chosen so that this stays below 1/8 cycle). A = |Xc|^2; mu = its mean.
// Cell (i, j), the quadrilateral of nodes (i, j) .. (i + 1, j + 1), gets the
// largest A / mu over the lags and bins its corners span (a max-pool of the
// map over the delay-Doppler box of the cell).
//
// Kernels:
//   k_coarse_init / k_coarse_geo / k_coarse_params   node lags and FDOAs
//       (double-float geometry, Eq. 3-10), their ranges per snapshot, the
//       map parameters;
//   chunk sums   by FFT correlation (k_chunk_spec and k_chunk_corr of dg_map.cu),
//       or for short chunks directly:
//   k_caf_lags   for one chunk and a tile of 896 lags, both sample windows sit in
//       shared memory; each thread slides a register window of y2 across 7
//       consecutive lags (7 is odd, so the lanes' strided reads hit distinct
//       banks): 7 x 7 complex FMAs per 14 loads;
//   k_caf_fold   the chunk DFT at the Q bins and |.|^2; deterministic partial
//       sums of A;
//   k_caf_pool   maxima of A over 8 consecutive lags, and mu per snapshot
//       (fixed-order sum);
//   k_coarse_backproject   the max-pool per cell.
#include <algorithm>
#include <cfloat>
#include <climits>

#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kCafR = 7;                          // lags per thread
constexpr int kCafThreads = 128;
constexpr int kCafTile = kCafR * kCafThreads;     // lags per k_caf_lags CTA
constexpr int kFoldWarps = 4;                     // warps of a k_caf_fold CTA
constexpr int kFoldBins = 16;                     // bin pairs per warp, at most
constexpr int kFoldRows = 16;                     // chunk pairs staged at a time
constexpr int kPoolLags = 8;                      // lags per pooled maximum

__device__ __forceinline__ float2 load_iq(const void *b, int fmt, int idx)
{
    if (fmt == DG_IQ_CI16) return IQ<DG_IQ_CI16>::load(b, idx);
    if (fmt == DG_IQ_CI8) return IQ<DG_IQ_CI8>::load(b, idx);
    return IQ<DG_IQ_C64>::load(b, idx);
}

// Order-preserving map of doubles onto unsigned 64-bit keys (and back).
__device__ __forceinline__ unsigned long long dkey(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double undkey(unsigned long long k)
{
    const unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)u);
}

__global__ void k_coarse_init(int *lmm, unsigned long long *nmm, int K)
{
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        lmm[2 * k] = INT_MAX;
        lmm[2 * k + 1] = INT_MIN;
        nmm[2 * k] = ~0ull;
        nmm[2 * k + 1] = 0ull;
    }
}

// Nodes of snapshot k = blockIdx.y, about eight per thread, the next one loaded
// while the current one is computed (228 -> 76 us for 20 snapshots of 513^2 nodes
// with that, the minima kept in FP32 and both receivers in packed operations; bound
// by the FP32 pipe): Eq. 3-10 in double-float
// arithmetic on the FP32 pipes (ranges to about 1e-7 m), the lag of Eq. 9
// (round half away from zero; decided by the FP64 expression where D lies
// within 1e-6 of a rounding boundary) and the FDOA rounded to FP32; block
// minima / maxima, then one atomic per warp.
__global__ void __launch_bounds__(256) k_coarse_geo(CoarseArgs a)
{
    const int k = blockIdx.y;
    dfl ed[12];
#pragma unroll
    for (int t = 0; t < 12; ++t) ed[t] = {__ldg(a.ephf + 24 * k + 2 * t), __ldg(a.ephf + 24 * k + 2 * t + 1)};
    const dfl fsc = {a.fsc_hi, a.fsc_lo}, ilf = {a.ilf_hi, a.ilf_lo};
    int lmin = INT_MAX, lmax = INT_MIN;
    float nmin = FLT_MAX, nmax = -FLT_MAX;
    const int64_t G = a.G;
    const float *xf = a.xyzf;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    float x[6];  // the next node, loaded one node ahead
    if (p < G)
#pragma unroll
        for (int e = 0; e < 6; ++e) x[e] = __ldg(xf + e * G + p);
    for (; p < G; p += step) {
        dfl D;
        float nu;
        const dfl nx = {x[0], x[1]}, ny = {x[2], x[3]}, nz = {x[4], x[5]};
        const int64_t pn = p + step < G ? p + step : p;
#pragma unroll
        for (int e = 0; e < 6; ++e) x[e] = __ldg(xf + e * G + pn);
        geometry_df(nx, ny, nz, ed, fsc, ilf, D, nu);
        int L;
        if (!round_df(D, L)) {
            double e[12], D64, nu64;
            for (int t = 0; t < 12; ++t) e[t] = a.eph[12 * k + t];
            geometry(a.xyz[p], a.xyz[G + p], a.xyz[2 * G + p], e, a.fs, a.lambda, D64, nu64);
            L = lag_of(D64, DG_DELAY_INTEGER);
        }
        a.lag[k * G + p] = L;
        a.nu[k * G + p] = nu;
        lmin = min(lmin, L);
        lmax = max(lmax, L);
        nmin = fminf(nmin, nu);
        nmax = fmaxf(nmax, nu);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        lmin = min(lmin, __shfl_xor_sync(0xffffffffu, lmin, d));
        lmax = max(lmax, __shfl_xor_sync(0xffffffffu, lmax, d));
        nmin = fminf(nmin, __shfl_xor_sync(0xffffffffu, nmin, d));
        nmax = fmaxf(nmax, __shfl_xor_sync(0xffffffffu, nmax, d));
    }
    if ((threadIdx.x & 31) == 0 && lmin <= lmax) {
        atomicMin(a.lmm + 2 * k, lmin);
        atomicMax(a.lmm + 2 * k + 1, lmax);
        atomicMin(a.nmm + 2 * k, dkey((double)nmin));
        atomicMax(a.nmm + 2 * k + 1, dkey((double)nmax));
    }
}

// The parameters of snapshot k = blockIdx.y (written by its first CTA), and the
// chunk DFT's factors: cos and sin of 2 pi d_j o_i M for the offset o_i = (nb - 1)
// / 2 - i of chunk pair i from the middle and half the distance d_j of bin pair j,
// two bin pairs a record (see k_caf_fold).
__global__ void __launch_bounds__(256) k_coarse_params(CoarseArgs a)
{
    const int k = blockIdx.y, H = a.Dpad / 2;
    const double lo = undkey(a.nmm[2 * k]), hi = undkey(a.nmm[2 * k + 1]);
    const double delta = a.Q > 1 ? __ddiv_rn(__dsub_rn(hi, lo), (double)(a.Q - 1)) : 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int l0 = a.lmm[2 * k], l1 = a.lmm[2 * k + 1];
        int nlag = (l1 >= l0) ? l1 - l0 + 1 : 0;
        if (nlag < 1 || nlag > a.nlag_cap) {
            atomicOr(a.err, ERR_LAG_RANGE);
            nlag = max(1, min(nlag, a.nlag_cap));
        }
        CoarseStep s;
        s.l0 = l0;
        s.nlag = nlag;
        s.nu_lo = lo;
        s.delta = delta;
        s.nu_c = __dmul_rn(0.5, __dadd_rn(lo, hi));
        s.mu = 0.0;
        a.st[k] = s;
        if (a.snap) {  // the correlation's lags, and its one Doppler node
            MapSnap m{};
            m.nuc = s.nu_c;
            m.L0 = l0;
            m.NL = nlag;
            a.snap[k] = m;
        }
    }
    const int nb = (a.steps[k].n + a.M - 1) / a.M, nh = (nb + 1) / 2;
    for (int64_t it = blockIdx.x * 256 + threadIdx.x; it < (int64_t)nh * H; it += gridDim.x * 256) {
        const int i = (int)(it / H), j = 2 * (int)(it % H);
        const double x = (0.5 * (nb - 1) - i) * (double)a.M;
        float s[2], c[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            double ph = (0.5 * (a.Q - 1) - (j + e)) * delta * x;
            ph = __dsub_rn(ph, floor(ph));
            sincospif(2.0f * (float)ph, &s[e], &c[e]);
        }
        a.turn[((size_t)k * a.nh_max + i) * H + j / 2] = make_float4(c[0], c[1], s[0], s[1]);
    }
}

// Chunk sums P_b(l) for chunk b = blockIdx.y of snapshot k = blockIdx.z and
// the lags t0 .. t0 + 895 (t0 = 896 blockIdx.x, relative to l0).
__global__ void __launch_bounds__(kCafThreads) k_caf_lags(CoarseArgs a)
{
    extern __shared__ float2 sm[];
    const int k = blockIdx.z, b = blockIdx.y;
    const CoarseStep st = a.st[k];
    const StepDesc sd = a.steps[k];
    const int t0 = blockIdx.x * kCafTile;
    const int M = a.M;
    const int64_t s0 = (int64_t)b * M;
    if (t0 >= st.nlag || s0 >= sd.n) return;
    float2 *as = sm;                    // [M + R]   y1 turned at nu_c
    float2 *cs = sm + M + kCafR;        // [M + T + 2R] y2 from sample s0 + l0 + t0
    for (int m = threadIdx.x; m < M + kCafR; m += kCafThreads) {
        const int64_t n = s0 + m;
        float2 v = make_float2(0.f, 0.f);
        if (m < M && n < sd.n) {
            const float2 y = load_iq(sd.y1, sd.fmt, (int)n);
            double ph = __dmul_rn(st.nu_c, (double)n);
            ph = __dsub_rn(ph, floor(ph));
            float sn, cn;
            sincospif(2.0f * (float)ph, &sn, &cn);
            v = make_float2(y.x * cn - y.y * sn, y.x * sn + y.y * cn);
        }
        as[m] = v;
    }
    const int64_t c0 = s0 + st.l0 + t0;
    for (int i = threadIdx.x; i < M + kCafTile + 2 * kCafR; i += kCafThreads) {
        const int64_t n = c0 + i;
        cs[i] = (n >= 0 && n < sd.n) ? load_iq(sd.y2, sd.fmt, (int)n) : make_float2(0.f, 0.f);
    }
    __syncthreads();

    const int base = kCafR * threadIdx.x;
    float accr[kCafR], acci[kCafR], w1r[kCafR], w1i[kCafR], w2r[kCafR], w2i[kCafR];
#pragma unroll
    for (int r = 0; r < kCafR; ++r) {
        accr[r] = acci[r] = 0.f;
        const float2 v = cs[base + r];
        w1r[r] = v.x;
        w1i[r] = v.y;
    }
    for (int m0 = 0; m0 < M; m0 += kCafR) {
#pragma unroll
        for (int r = 0; r < kCafR; ++r) {
            const float2 v = cs[m0 + kCafR + base + r];
            w2r[r] = v.x;
            w2i[r] = v.y;
        }
#pragma unroll
        for (int s = 0; s < kCafR; ++s) {
            const float2 av = as[m0 + s];
#pragma unroll
            for (int r = 0; r < kCafR; ++r) {
                const int q = r + s;
                const float vr = q < kCafR ? w1r[q] : w2r[q - kCafR];
                const float vi = q < kCafR ? w1i[q] : w2i[q - kCafR];
                // av * conj(v)
                accr[r] = fmaf(av.x, vr, fmaf(av.y, vi, accr[r]));
                acci[r] = fmaf(av.y, vr, fmaf(-av.x, vi, acci[r]));
            }
        }
#pragma unroll
        for (int r = 0; r < kCafR; ++r) {
            w1r[r] = w2r[r];
            w1i[r] = w2i[r];
        }
    }
    float2 *Pk = a.P + ((size_t)k * a.nb_max + b) * a.nlag_cap;
#pragma unroll
    for (int r = 0; r < kCafR; ++r) {
        const int t = t0 + base + r;
        if (t < st.nlag) Pk[t] = make_float2(accr[r], acci[r]);
    }
}

// Whether lag L's sum reads a sample that is not finite. Every lag's does where
// y1 holds one (zeros of y2 included: 0 x NaN); y2's index runs from L over the
// nx samples that the direct kernel sums.
__device__ __forceinline__ bool caf_bad(int4 b, int L, int nx)
{
    if (b.y >= 0) return true;
    return b.w >= 0 && (L >= 0 ? b.w >= L : b.z < nx + L);
}

// Xc at the Q bins for the CTA's lags of snapshot k = blockIdx.y: a warp takes
// 32 lags and 2 H bin pairs. The bins lie symmetrically around nu_c and the
// chunks around their middle, and a unit phase per bin drops out of |.|^2: bins
// nu_c +- d and chunks at offsets +- o share
//     C = sum cos(2 pi d o M) (P_+ + P_-),   S = sum sin(2 pi d o M) (P_+ - P_-),
//     Xc(nu_c +- d) = C +- j S,
// 4 real FMAs for 2 bins x 2 chunks where the complex products take 16. FP32
// pipe; the factors (k_coarse_params) and the chunk pairs' sums and differences come
// from shared memory, two bin pairs per packed FMA. 20 snapshots of 4192 lags,
// 128 chunks and 40 bins: 254 -> 34 us. A = |Xc|^2, lags fastest, and the CTA's
// sum of A (in a fixed order). QW of the CTA's warps lie along the bins.
__device__ __forceinline__ void fma2_to(float2 &c, float2 a, float2 b)
{
    unsigned long long r, x, y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(r));
}

__device__ __forceinline__ void cp_async8z(void *dst, const void *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(in ? 8u : 0u)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int QW, int H> __global__ void __launch_bounds__(32 * kFoldWarps) k_caf_fold(CoarseArgs a)
{
    constexpr int LW = kFoldWarps / QW, NL = 32 * LW, T = 32 * kFoldWarps;
    extern __shared__ __align__(16) unsigned char fold_sm[];
    float4 *s_w = reinterpret_cast<float4 *>(fold_sm);                   // [2][rows][QW H] cos, sin of two bin pairs
    float2 *s_p = reinterpret_cast<float2 *>(s_w + 2 * kFoldRows * QW * H);  // [2][rows][2][NL] the pair's chunks
    __shared__ double red[kFoldWarps];
    const int k = blockIdx.y, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const CoarseStep st = a.st[k];
    const int lt0 = blockIdx.x * NL, part = blockIdx.z * gridDim.x + blockIdx.x, parts = gridDim.x * gridDim.z;
    if (lt0 >= st.nlag) {
        if (t == 0) a.part[(size_t)k * parts + part] = 0.0;
        return;
    }
    const int N = a.steps[k].n, nb = (N + a.M - 1) / a.M, nh = (nb + 1) / 2, ns = (nh + kFoldRows - 1) / kFoldRows;
    const int wq = warp % QW, wl = warp / QW;
    const int j0 = (blockIdx.z * QW + wq) * 2 * H, nq2 = (a.Q + 1) / 2;  // bin pairs, the middle bin one of them
    const float2 *Pk = a.P + (size_t)k * a.nb_max * a.nlag_cap;
    const float4 *W = a.turn + (size_t)k * a.nh_max * (a.Dpad / 2) + blockIdx.z * QW * H;
    auto stage = [&](int g) {  // chunk pairs g kFoldRows .. , asynchronously
        if (g < ns) {
            const int i0 = g * kFoldRows, nr = min(kFoldRows, nh - i0);
            for (int x = t; x < nr * 2 * NL; x += T) {
                const int r = x / (2 * NL), h = x / NL & 1, l = lt0 + x % NL, b = i0 + r, bh = nb - 1 - b;
                // the middle chunk of an odd number has no partner (and sin = 0)
                const bool in = l < st.nlag && (h || bh != b);
                cp_async8z(s_p + (g & 1) * kFoldRows * 2 * NL + x, in ? Pk + (size_t)(h ? bh : b) * a.nlag_cap + l : Pk, in);
            }
            for (int x = t; x < nr * QW * H; x += T)
                cp_async16(s_w + (g & 1) * kFoldRows * QW * H + x,
                           W + (size_t)(i0 + x / (QW * H)) * (a.Dpad / 2) + x % (QW * H));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 cr[H], ci[H], sr[H], si[H];
#pragma unroll
    for (int h = 0; h < H; ++h) cr[h] = ci[h] = sr[h] = si[h] = make_float2(0.f, 0.f);
    stage(0);
    for (int g = 0; g < ns; ++g) {
        stage(g + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        if (j0 < nq2) {
            const int nr = min(kFoldRows, nh - g * kFoldRows);
            const float2 *p_s = s_p + (g & 1) * kFoldRows * 2 * NL + 32 * wl + lane;
            const float4 *w_s = s_w + (g & 1) * kFoldRows * QW * H + wq * H;
            for (int r = 0; r < nr; ++r, p_s += 2 * NL, w_s += QW * H) {
                const float2 lo = p_s[0], hi = p_s[NL];
                const float2 ur = make_float2(hi.x + lo.x, hi.x + lo.x), ui = make_float2(hi.y + lo.y, hi.y + lo.y);
                const float2 vr = make_float2(hi.x - lo.x, hi.x - lo.x), vi = make_float2(hi.y - lo.y, hi.y - lo.y);
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const float4 w = w_s[h];
                    const float2 c = make_float2(w.x, w.y), n = make_float2(w.z, w.w);
                    fma2_to(cr[h], c, ur);
                    fma2_to(ci[h], c, ui);
                    fma2_to(sr[h], n, vr);
                    fma2_to(si[h], n, vi);
                }
            }
        }
        __syncthreads();  // the buffer is free for stage g + 2
    }
    const int l = lt0 + 32 * wl + lane;
    double sum = 0.0;
    if (l < st.nlag && j0 < nq2) {
        const bool bad = a.bad && caf_bad(reinterpret_cast<const int4 *>(a.bad)[k], st.l0 + l,
                                          (nb - 1) * a.M + (a.M + kCafR - 1) / kCafR * kCafR);
        float *Ak = a.A + (size_t)k * a.Q * a.nlag_cap + l;
#pragma unroll
        for (int z = 0; z < 2 * H; ++z) {
            const int j = j0 + z;
            if (j >= nq2) continue;
            const float c0 = z & 1 ? cr[z / 2].y : cr[z / 2].x, c1 = z & 1 ? ci[z / 2].y : ci[z / 2].x;
            const float s0 = z & 1 ? sr[z / 2].y : sr[z / 2].x, s1 = z & 1 ? si[z / 2].y : si[z / 2].x;
            float up = fmaf(c0 - s1, c0 - s1, (c1 + s0) * (c1 + s0));
            float dn = fmaf(c0 + s1, c0 + s1, (c1 - s0) * (c1 - s0));
            if (bad) up = dn = __int_as_float(0x7fffffff);
            Ak[(size_t)(a.Q - 1 - j) * a.nlag_cap] = up;
            sum += (double)up;
            if (2 * j != a.Q - 1) {
                Ak[(size_t)j * a.nlag_cap] = dn;
                sum += (double)dn;
            }
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lane == 0) red[warp] = sum;
    __syncthreads();
    if (t == 0) {
        double s = 0.0;
        for (int w = 0; w < kFoldWarps; ++w) s += red[w];
        a.part[(size_t)k * parts + part] = s;
    }
}

// Maxima over kPoolLags lags from each lag on (clipped at the last), per bin;
// the first CTA of a snapshot also sums mu. A cell's box then takes one or two
// loads per bin where its lags would take a dozen.
__global__ void __launch_bounds__(256) k_caf_pool(CoarseArgs a, int parts)
{
    __shared__ float s_a[256 + kPoolLags];
    __shared__ double red[8];
    const int k = blockIdx.z, q = blockIdx.y, l0 = blockIdx.x * 256, t = threadIdx.x;
    const int nlag = a.st[k].nlag;
    if (blockIdx.x == 0 && q == 0) {
        double s = 0.0;
        for (int i = t; i < parts; i += 256) s += a.part[(size_t)k * parts + i];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if ((t & 31) == 0) red[t >> 5] = s;
        __syncthreads();
        if (t == 0) {
            double m = 0.0;
            for (int w = 0; w < 8; ++w) m += red[w];
            a.st[k].mu = m / ((double)nlag * (double)a.Q);
        }
    }
    if (l0 >= nlag) return;
    const float *A = a.A + ((size_t)k * a.Q + q) * a.nlag_cap;
    for (int x = t; x < 256 + kPoolLags; x += 256) s_a[x] = l0 + x < nlag ? A[l0 + x] : 0.f;
    __syncthreads();
    float m = s_a[t];
#pragma unroll
    for (int x = 1; x < kPoolLags; ++x) m = fmaxf(m, s_a[t + x]);
    if (l0 + t < nlag) a.pool[((size_t)k * a.Q + q) * a.nlag_cap + l0 + t] = m;
}

// A with the bins fastest, [nlag_cap][Q] per snapshot (dg_coarse_inspect).
__global__ void __launch_bounds__(256) k_caf_transpose(const float *__restrict__ A, float *__restrict__ out, int Q, int cap)
{
    __shared__ float s[32][33];
    const int k = blockIdx.z, l0 = blockIdx.x * 32, q0 = blockIdx.y * 32, x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (q0 + y < Q && l0 + x < cap) s[y][x] = A[((size_t)k * Q + q0 + y) * cap + l0 + x];
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (l0 + y < cap && q0 + x < Q) out[((size_t)k * cap + l0 + y) * Q + q0 + x] = s[x][y];
}

// (v - lo) / delta of FP32 FDOAs v and lo in bins, rounded down or up. In FP32
// the quotient is off by under 4 2^-24 of itself (Q <= 256 bins: 6.1e-5);
// within 1e-4 of an integer the FP64 expression decides.
__device__ __forceinline__ int bin_of(float v, const CoarseStep &st, float lo, float inv, bool up)
{
    const float x = (v - lo) * inv, r = rintf(x);
    if (fabsf(x - r) < 1e-4f) {
        const double d = __ddiv_rn(__dsub_rn((double)v, st.nu_lo), st.delta);
        return (int)(up ? ceil(d) : floor(d));
    }
    return (int)(up ? ceilf(x) : floorf(x));
}

// Cells of column j (one thread) and kBackRows rows of snapshot k =
// blockIdx.z: a cell's box of A through the pooled maxima, the corners of a row
// kept for the next one. FP32 except next to a bin edge: the FP64 quotients and
// the division by mu of every cell were bound by the FP64 units, the loads of a
// box with the bins fastest by L1 (432 -> 65 us for 20 snapshots of 512^2 cells).
constexpr int kBackRows = 8;
__global__ void __launch_bounds__(128) k_coarse_backproject(CoarseArgs a)
{
    const int k = blockIdx.z;
    const CoarseStep st = a.st[k];
    const int Q = a.Q;
    const int nlon = a.nlon, ncol = nlon - 1, nrow = a.nlat - 1;
    const int64_t ncell = (int64_t)nrow * ncol;
    const int *lag = a.lag + (size_t)k * a.G;
    const float *nu = a.nu + (size_t)k * a.G;
    const float *Ak = a.A + (size_t)k * a.nlag_cap * Q, *Bk = a.pool + (size_t)k * a.nlag_cap * Q;
    const float lo = (float)st.nu_lo, inv = (float)(1.0 / st.delta);
    const double im = 1.0 / st.mu;
    const float im_hi = (float)im, im_lo = (float)(im - (double)im_hi);
    const bool fast = im_hi > 1e-30f && im_hi < 1e30f;
    for (int j = blockIdx.x * 128 + threadIdx.x; j < ncol; j += gridDim.x * 128)
        for (int i0 = blockIdx.y * kBackRows; i0 < nrow; i0 += gridDim.y * kBackRows) {
            const int64_t p0 = (int64_t)i0 * nlon + j;
            int l0 = __ldg(lag + p0), l1 = __ldg(lag + p0 + 1);
            float v0 = __ldg(nu + p0), v1 = __ldg(nu + p0 + 1);
            int ll = min(l0, l1), lh = max(l0, l1);
            float vl = fminf(v0, v1), vh = fmaxf(v0, v1);
#pragma unroll 2
            for (int r = 0; r < kBackRows && i0 + r < nrow; ++r) {
                const int64_t p = p0 + (int64_t)(r + 1) * nlon;
                l0 = __ldg(lag + p);
                l1 = __ldg(lag + p + 1);
                v0 = __ldg(nu + p);
                v1 = __ldg(nu + p + 1);
                const int la = max(0, min(ll, min(l0, l1)) - st.l0), lb = min(st.nlag - 1, max(lh, max(l0, l1)) - st.l0);
                const float vmin = fminf(vl, fminf(v0, v1)), vmax = fmaxf(vh, fmaxf(v0, v1));
                ll = min(l0, l1);
                lh = max(l0, l1);
                vl = fminf(v0, v1);
                vh = fmaxf(v0, v1);
                int qa = 0, qb = Q - 1;
                if (st.delta > 0.0) {
                    qa = max(0, bin_of(vmin, st, lo, inv, false));
                    qb = min(Q - 1, bin_of(vmax, st, lo, inv, true));
                }
                float m = 0.f;
                const int len = lb - la + 1;
                const float *row = (len >= kPoolLags ? Bk : Ak) + (int64_t)qa * a.nlag_cap + la;
                const int step = len >= kPoolLags ? kPoolLags : 1, last = len - step;
                for (int q = qa; q <= qb; ++q, row += a.nlag_cap) {
                    for (int t = 0; t < last; t += step) m = fmaxf(m, __ldg(row + t));
                    if (last >= 0) m = fmaxf(m, __ldg(row + last));
                }
                // m / mu: m times the reciprocal in two words
                const float h = m * im_hi;
                const float v = h + fmaf(m, im_lo, fmaf(m, im_hi, -h));
                a.maps[(size_t)k * ncell + (int64_t)(i0 + r) * ncol + j] =
                    st.mu > 0.0 ? (fast && isfinite(h) ? v : (float)((double)m / st.mu)) : 0.f;
            }
        }
}

unsigned blocks_for(int64_t n, int per, int cap)
{
    int64_t b = (n + per - 1) / per;
    return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

// Warps of a CTA along the bins, and the bin pairs of one (an even number: the
// pairs in equal parts, so that a map of 40 bins leaves none of them idle).
static int fold_qw(int Q) { return (Q + 1) / 2 <= kFoldBins ? 1 : (Q + 1) / 2 <= 2 * kFoldBins ? 2 : 4; }
static int fold_pairs(int Q)
{
    const int qw = fold_qw(Q), p = std::min(kFoldBins, ((Q + 1) / 2 + qw - 1) / qw);
    return p <= 8 ? 8 : p <= 10 ? 10 : p <= 12 ? 12 : 16;
}
int coarse_parts(int nlag_cap, int Q)
{
    const int nl = 32 * (kFoldWarps / fold_qw(Q)), nj = fold_pairs(Q) * fold_qw(Q);
    return (nlag_cap + nl - 1) / nl * (((Q + 1) / 2 + nj - 1) / nj);
}
int coarse_dpad(int Q)
{
    const int nj = fold_pairs(Q) * fold_qw(Q);
    return ((Q + 1) / 2 + nj - 1) / nj * nj;
}

template <int QW, int H> static cudaError_t launch_fold_h(const CoarseArgs &a, cudaStream_t s)
{
    const unsigned nl = 32 * (kFoldWarps / QW), nj = 2 * H * QW;
    const size_t smem = kFoldRows * (sizeof(float4) * 2 * nj / 2 + sizeof(float2) * 4 * nl);
    const cudaError_t e = cudaFuncSetAttribute(k_caf_fold<QW, H>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_caf_fold<QW, H><<<dim3((a.nlag_cap + nl - 1) / nl, a.K, ((a.Q + 1) / 2 + nj - 1) / nj), 32 * kFoldWarps, smem, s>>>(a);
    return cudaGetLastError();
}
template <int QW> static cudaError_t launch_fold(const CoarseArgs &a, cudaStream_t s)
{
    switch (fold_pairs(a.Q)) {
    case 8: return launch_fold_h<QW, 4>(a, s);
    case 10: return launch_fold_h<QW, 5>(a, s);
    case 12: return launch_fold_h<QW, 6>(a, s);
    default: return launch_fold_h<QW, 8>(a, s);
    }
}

cudaError_t launch_coarse(const CoarseArgs &a, const MapArgs *fft, cudaStream_t s, int *launches)
{
    cudaError_t e;
    k_coarse_params<<<dim3(blocks_for((int64_t)a.nh_max * a.Dpad / 2, 256, 152 * 8), a.K), 256, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (fft) {
        if ((e = launch_chunk_sums(*fft, s, launches)) != cudaSuccess) return e;
    } else {
        const size_t lag_smem = sizeof(float2) * (2 * (size_t)a.M + kCafTile + 3 * kCafR);
        if (lag_smem > 48 * 1024) {
            e = cudaFuncSetAttribute(k_caf_lags, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lag_smem);
            if (e != cudaSuccess) return e;
        }
        k_caf_lags<<<dim3((a.nlag_cap + kCafTile - 1) / kCafTile, a.nb_max, a.K), kCafThreads, lag_smem, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        ++*launches;
    }
    const int qw = fold_qw(a.Q);
    e = qw == 1 ? launch_fold<1>(a, s) : qw == 2 ? launch_fold<2>(a, s) : launch_fold<4>(a, s);
    if (e != cudaSuccess) return e;
    k_caf_pool<<<dim3((a.nlag_cap + 255) / 256, a.Q, a.K), 256, 0, s>>>(a, coarse_parts(a.nlag_cap, a.Q));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_coarse_backproject<<<dim3(blocks_for(a.nlon - 1, 128, 65535), blocks_for(a.nlat - 1, kBackRows, 65535), a.K), 128, 0,
                           s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *launches += 4;
    return cudaSuccess;
}

// The nodes' lags and FDOAs and their ranges: needs no shape of the maps.
cudaError_t launch_coarse_geo(const CoarseArgs &a, cudaStream_t s, int *launches)
{
    cudaError_t e;
    k_coarse_init<<<1, 64, 0, s>>>(a.lmm, a.nmm, a.K);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_coarse_geo<<<dim3(blocks_for(a.G, 256, 152 * 3 * 4 / a.K + 1), a.K), 256, 0, s>>>(a);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_coarse_transpose(const float *A, float *out, int K, int Q, int nlag_cap, cudaStream_t s)
{
    k_caf_transpose<<<dim3((nlag_cap + 31) / 32, (Q + 31) / 32, K), 256, 0, s>>>(A, out, Q, nlag_cap);
    return cudaGetLastError();
}

}  // namespace dg
