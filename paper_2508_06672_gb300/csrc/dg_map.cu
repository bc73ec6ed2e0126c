// dg_map.cu -- Eq. 11 from delay-Doppler maps: the chunked-DFT evaluation
// (DG_ALGO_CDFT) of a grid of many nodes with FP32 arithmetic.
//
// Every candidate c of snapshot k needs the cross-ambiguity function
//     X(l, nu) = sum_n y1[n] conj(y2[n + l]) e^{j 2 pi nu (n - N/2)}
// at its own integer lag l (Eq. 9) and FDOA nu (Eq. 10), up to the unit phase
// e^{j pi nu N} that |.| removes. The grid's lags and FDOAs cover a narrow
// rectangle, so X is tabulated once per snapshot on every lag of it and on Q
// Doppler bins, and each candidate interpolates the table in Doppler.
//
//   spec    FFT (n points) of each y2 window of a block of Mb samples, and
//           the block's phases e^{j 2 pi nu_q t_c} at the bins;
//   corr    per (block c, Doppler node p): the block of y1 turned at nu_p,
//           its FFT times the window's conjugate spectrum, and a second FFT:
//           U[c][p][l] = sum_m y1[cMb + m] e^{j 2 pi nu_p (m - Mb/2)}
//           conj(y2[cMb + m + l]) for all lags of a tile at once. Over one
//           block X is smooth in nu (its phase turns by less than one
//           or two cycles across the band), so P Chebyshev nodes nu_p fix it;
//   expand  X[q][l] = sum_c e^{j 2 pi nu_q t_c} sum_p T_p(nu_q) U[c][p][l],
//           T_p the nodes' Lagrange polynomials at the bins, t_c the block's
//           centre relative to the capture's;
//   lookup  per candidate, snapshots in order: geometry, six bins around its
//           FDOA (Lagrange), |.|^2 or |.|, summed in a register.
//
// A correlation of n lags through two FFTs costs about 10 n log2 n flop where
// the contraction of dg_cdft_mma.cu costs 512 flop per (lag, sample): the
// 4001^2-node, 50-snapshot workload needs 0.1 TFLOP for its tables instead of
// 18. The lookup gathers from tables stored lag-fastest: neighbouring nodes of
// a grid row have neighbouring lags and nearly the same FDOA, so a warp's
// loads fall into a few cache lines and nothing has to be sorted.
//
// FFT: the Stockham autosort form (Govindaraju et al., "High performance
// discrete Fourier transforms on graphics processors", 2008): 16 points per
// thread, radix-16 passes in registers with one shared-memory exchange
// between passes (one pad element per 16 keeps the stride-16 stores of the
// first exchange free of bank conflicts), the remaining radix last, so input
// and output have the same distribution (element t + T e in thread t).
#include "dg_internal.cuh"

namespace dg {
namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// Two FP32 FMAs in one instruction (Blackwell's packed form): half the issue
// slots of the same arithmetic.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
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

__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Sums and differences of complex pairs in one instruction (a - b as a + b (-1),
// exact), where both parts take the same sign and place.
__device__ __forceinline__ float2 cadd(float2 a, float2 b)
{
    unsigned long long r, x, y;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(r));
    return d;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return fma2(b, make_float2(-1.f, -1.f), a); }

// e^{j 2 pi f x} for a frequency f = hi + lo (cycles per sample) and an
// integer-valued x, |x| < 2^24.
__device__ __forceinline__ float2 cis_df(float hi, float lo, float x)
{
    float s, c;
    sincospif(2.0f * (frac_mul(hi, x) + lo * x), &s, &c);
    return make_float2(c, s);
}

// Forward DFTs of 2, 4, 8 and 16 points in registers; output k of fft16 is
// v[4 (k % 4) + k / 4], of fft8 v[2 (k % 4) + k / 4].
__device__ __forceinline__ void fft2(float2 &a, float2 &b)
{
    const float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
__device__ __forceinline__ void fft4(float2 &a, float2 &b, float2 &c, float2 &d)
{
    const float2 s = cadd(a, c), t = csub(a, c), u = cadd(b, d), w = csub(b, d);
    a = cadd(s, u);
    b = make_float2(t.x + w.y, t.y - w.x);  // t - j w
    c = csub(s, u);
    d = make_float2(t.x - w.y, t.y + w.x);
}
constexpr float kC8 = 0.70710678118654752f, kC16 = 0.92387953251128674f, kS16 = 0.38268343236508977f;
__device__ __forceinline__ float2 rot8(float2 a)  // times e^{-j pi / 4}
{
    return make_float2(kC8 * (a.x + a.y), kC8 * (a.y - a.x));
}
__device__ __forceinline__ float2 rotj(float2 a) { return make_float2(a.y, -a.x); }  // times -j

__device__ __forceinline__ void fft16(float2 (&v)[16])
{
#pragma unroll
    for (int a = 0; a < 4; ++a) fft4(v[a], v[a + 4], v[a + 8], v[a + 12]);
    // v[a + 4 k] times e^{-j 2 pi a k / 16}
    const float2 w1 = make_float2(kC16, -kS16), w3 = make_float2(kS16, -kC16);
    v[5] = cmul(v[5], w1);
    v[6] = rot8(v[6]);
    v[7] = cmul(v[7], w3);
    v[9] = rot8(v[9]);
    v[10] = rotj(v[10]);
    v[11] = rotj(rot8(v[11]));
    v[13] = cmul(v[13], w3);
    v[14] = rotj(rot8(v[14]));
    v[15] = cmul(v[15], make_float2(-kC16, kS16));
#pragma unroll
    for (int k = 0; k < 4; ++k) fft4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}
__device__ __forceinline__ constexpr int pos16(int k) { return 4 * (k & 3) + (k >> 2); }

// The last pass of radix R < 16: 16 / R butterflies of elements i + r (16 / R).
template <int R> __device__ __forceinline__ void fft_small(float2 (&v)[16])
{
    constexpr int S = 16 / R;
#pragma unroll
    for (int i = 0; i < S; ++i) {
        if constexpr (R == 2) {
            fft2(v[i], v[i + S]);
        } else if constexpr (R == 4) {
            fft4(v[i], v[i + S], v[i + 2 * S], v[i + 3 * S]);
        } else {
            float2 e0 = v[i], e1 = v[i + 2 * S], e2 = v[i + 4 * S], e3 = v[i + 6 * S];
            float2 o0 = v[i + S], o1 = v[i + 3 * S], o2 = v[i + 5 * S], o3 = v[i + 7 * S];
            fft4(e0, e1, e2, e3);
            fft4(o0, o1, o2, o3);
            o1 = rot8(o1);
            o2 = rotj(o2);
            o3 = rotj(rot8(o3));
            v[i] = cadd(e0, o0);
            v[i + S] = cadd(e1, o1);
            v[i + 2 * S] = cadd(e2, o2);
            v[i + 3 * S] = cadd(e3, o3);
            v[i + 4 * S] = csub(e0, o0);
            v[i + 5 * S] = csub(e1, o1);
            v[i + 6 * S] = csub(e2, o2);
            v[i + 7 * S] = csub(e3, o3);
        }
    }
}

__device__ __forceinline__ int pad16(int i) { return i + (i >> 4); }

// v[e] times w^{e idx} of a radix-R butterfly, w = e^{-j 2 pi / n}: the
// powers 1, 2, 4, 8 from the table, the others as one product each.
template <int R, int STRIDE>
__device__ __forceinline__ void twiddle(float2 *v, const float2 *__restrict__ tw, int idx)
{
    const float2 w1 = __ldg(tw + idx);
    v[STRIDE] = cmul(v[STRIDE], w1);
    if constexpr (R >= 4) {
        const float2 w2 = __ldg(tw + 2 * idx), w3 = cmul(w1, w2);
        v[2 * STRIDE] = cmul(v[2 * STRIDE], w2);
        v[3 * STRIDE] = cmul(v[3 * STRIDE], w3);
        if constexpr (R >= 8) {
            const float2 w4 = __ldg(tw + 4 * idx);
            v[4 * STRIDE] = cmul(v[4 * STRIDE], w4);
            v[5 * STRIDE] = cmul(v[5 * STRIDE], cmul(w4, w1));
            v[6 * STRIDE] = cmul(v[6 * STRIDE], cmul(w4, w2));
            v[7 * STRIDE] = cmul(v[7 * STRIDE], cmul(w4, w3));
            if constexpr (R >= 16) {
                const float2 w8 = __ldg(tw + 8 * idx), w12 = cmul(w8, w4);
                v[8] = cmul(v[8], w8);
                v[9] = cmul(v[9], cmul(w8, w1));
                v[10] = cmul(v[10], cmul(w8, w2));
                v[11] = cmul(v[11], cmul(w8, w3));
                v[12] = cmul(v[12], w12);
                v[13] = cmul(v[13], cmul(w12, w1));
                v[14] = cmul(v[14], cmul(w12, w2));
                v[15] = cmul(v[15], cmul(w12, w3));
            }
        }
    }
}

// n = 2^LOGN point forward DFT of the CTA's n / 16 threads, in place; s holds
// pad16(n) elements. Enters and leaves with s free (a barrier before each use).
template <int LOGN> __device__ __forceinline__ void fft_cta(float2 (&v)[16], float2 *s, const float2 *__restrict__ tw)
{
    constexpr int n = 1 << LOGN, T = n / 16, full = LOGN / 4, rest = LOGN % 4;
    const int t = threadIdx.x;
#pragma unroll
    for (int p = 0; p < full; ++p) {
        const int Ns = 1 << (4 * p);
        if (p > 0) twiddle<16, 1>(v, tw, (t & (Ns - 1)) << (LOGN - 4 * p - 4));
        fft16(v);
        if (p + 1 < full || rest) {
            const int d = ((t >> (4 * p)) << (4 * p + 4)) + (t & (Ns - 1));
            __syncthreads();
#pragma unroll
            for (int r = 0; r < 16; ++r) s[pad16(d + r * Ns)] = v[pos16(r)];
            __syncthreads();
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = s[pad16(t + e * T)];
        } else {
            float2 u[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) u[r] = v[pos16(r)];
#pragma unroll
            for (int r = 0; r < 16; ++r) v[r] = u[r];
        }
    }
    if constexpr (rest > 0) {
        constexpr int R = 1 << rest, S = 16 / R;
#pragma unroll
        for (int i = 0; i < S; ++i) twiddle<R, S>(v + i, tw, t + i * T);  // Ns = n / R: index j
        fft_small<R>(v);
    }
}

// Sample i of a capture as FP32; a value that is not finite counts as zero
// (only c64 captures can hold one; its lags are flagged apart).
__device__ __forceinline__ float2 load_sample(const void *b, int fmt, int i)
{
    if (fmt == DG_IQ_CI16) return IQ<DG_IQ_CI16>::load(b, i);
    if (fmt == DG_IQ_CI8) return IQ<DG_IQ_CI8>::load(b, i);
    const float2 v = IQ<DG_IQ_C64>::load(b, i);
    return isfinite(v.x) && isfinite(v.y) ? v : make_float2(0.f, 0.f);
}

}  // namespace

__global__ void k_map_twiddles(float2 *tw, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float s, c;
    sincospif(-2.0f * (float)i / (float)n, &s, &c);  // i / n is exact
    tw[i] = make_float2(c, s);
}

// First and last sample of each capture that is not finite (c64 captures).
__global__ void k_map_bad_init(int *bad, int S)
{
    for (int i = threadIdx.x; i < S; i += blockDim.x) {
        bad[4 * i] = bad[4 * i + 2] = 0x7fffffff;
        bad[4 * i + 1] = bad[4 * i + 3] = -1;
    }
}
__global__ void __launch_bounds__(256) k_map_bad(MapArgs a)
{
    const int s = blockIdx.y, r = blockIdx.z;
    const StepDesc sd = a.sd[s];
    if (sd.fmt != DG_IQ_C64) return;
    const float2 *y = reinterpret_cast<const float2 *>(r ? sd.y2 : sd.y1);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < sd.n; i += gridDim.x * blockDim.x) {
        const float2 v = __ldg(y + i);
        if (!(isfinite(v.x) && isfinite(v.y))) {
            atomicMin(a.bad + 4 * s + 2 * r, i);
            atomicMax(a.bad + 4 * s + 2 * r + 1, i);
        }
    }
}

template <int LOGN> __global__ void __launch_bounds__((1 << LOGN) / 16) k_map_spec(MapArgs a)
{
    constexpr int n = 1 << LOGN, T = n / 16;
    extern __shared__ __align__(16) float2 sm[];
    const int t = threadIdx.x, c = blockIdx.x, tile = blockIdx.y, s = blockIdx.z;
    const StepDesc sd = a.sd[s % a.ksd];
    const MapSnap ms = a.snap[s];
    if ((int64_t)c * a.Mb >= sd.n || tile * a.LT >= ms.NL) return;
    if (tile == 0) {  // the block's phases at the bins
        const double tc = (double)((int64_t)c * a.Mb + a.Mb / 2 - sd.n / 2);
        for (int q = t; q < a.Q; q += T) {
            const double ph = (ms.nu0 + q * ms.delta) * tc;
            float sn, cs;
            sincospif((float)(2.0 * (ph - floor(ph))), &sn, &cs);
            a.phase[((size_t)s * a.Cmax + c) * a.Q + q] = make_float2(cs, sn);
        }
    }
    const int64_t i0 = (int64_t)c * a.Mb + ms.L0 + (int64_t)tile * a.LT;
    float2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int64_t i = i0 + t + T * e;
        v[e] = i >= 0 && i < sd.n ? load_sample(sd.y2, sd.fmt, (int)i) : make_float2(0.f, 0.f);
    }
    fft_cta<LOGN>(v, sm, a.tw);
    float2 *F = a.F2 + (((size_t)s * a.ntile + tile) * a.Cmax + c) * n + t;
#pragma unroll
    for (int e = 0; e < 16; ++e) F[T * e] = v[e];
}

template <int LOGN>
__global__ void __launch_bounds__((1 << LOGN) / 16, LOGN == 14 ? 1 : LOGN == 13 ? 2 : 1024 * 16 / (1 << LOGN)) k_map_corr(MapArgs a)
{
    constexpr int n = 1 << LOGN, T = n / 16;
    extern __shared__ __align__(16) float2 sm[];
    __shared__ float2 s_step[16];
    __shared__ float s_nu[2];
    const int t = threadIdx.x, p = blockIdx.x % a.P, c = blockIdx.x / a.P, tile = blockIdx.y, s = blockIdx.z;
    const StepDesc sd = a.sd[s % a.ksd];
    const MapSnap ms = a.snap[s];
    const int64_t n0 = (int64_t)c * a.Mb;
    if (n0 >= sd.n || tile * a.LT >= ms.NL) return;
    // the node's frequency and the phasors of the thread's samples,
    // e^{j 2 pi nu_p (t - Mb/2)} e^{j 2 pi nu_p T e}
    if (t == 0) {
        const double nup = ms.nuc + ms.halfw * a.xnode[p];
        s_nu[0] = (float)nup;
        s_nu[1] = (float)(nup - (double)s_nu[0]);
    }
    __syncthreads();
    const float nh = s_nu[0], nl = s_nu[1];
    if (t < 16) s_step[t] = cis_df(nh, nl, (float)(T * t));
    const float2 base = cis_df(nh, nl, (float)(t - a.Mb / 2));
    __syncthreads();
    const int len = (int)min((int64_t)a.Mb, sd.n - n0);
    float2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int m = t + T * e;
        v[e] = m < len ? load_sample(sd.y1, sd.fmt, (int)(n0 + m)) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = cmul(v[e], cmul(base, s_step[e]));
    const float2 *F = a.F2 + (((size_t)s * a.ntile + tile) * a.Cmax + c) * n + t;
    constexpr float inv = 1.0f / (float)n;
    // both transforms through one copy of the code: inlined twice, the
    // compiler keeps the first one's twiddles in registers for the second
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        fft_cta<LOGN>(v, sm, a.tw);
        if (pass == 0) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float2 f = __ldg(F + T * e);
                v[e] = make_float2(fmaf(v[e].x, f.x, v[e].y * f.y) * inv, fmaf(v[e].y, f.x, -v[e].x * f.y) * inv);
            }
        }
    }
    float2 *U = a.U + (((size_t)s * a.Cmax + c) * a.P + p) * a.NLpad;
    const int l0 = tile * a.LT, nl_t = min(a.LT, ms.NL - l0);
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int l = t + T * e;
        if (l < nl_t) U[l0 + l] = v[e];
    }
}

// Chunk sums of the coarse maps (dg_coarse.cu): for each chunk c of Mb = M samples
// and lag l, sum_m y1[cM + m] e^{j 2 pi nuc (cM + m)} conj(y2[cM + m + l]). The
// windows of y2 start M samples apart and the lag tiles LT = n - M apart, a
// multiple of M (both powers of two): window w = c + tile LT / M serves every
// chunk and tile of that sum, so a snapshot takes Cmax + nwin forward transforms
// and one inverse per (chunk, tile), where a window and a turned chunk per (chunk,
// tile) took three. F2: [S][Cmax + nwin][n].
template <int LOGN> __global__ void __launch_bounds__((1 << LOGN) / 16) k_chunk_spec(MapArgs a)
{
    constexpr int n = 1 << LOGN, T = n / 16;
    extern __shared__ __align__(16) float2 sm[];
    __shared__ float2 s_step[16];
    const int t = threadIdx.x, s = blockIdx.y, c = blockIdx.x, w = c - a.Cmax, hop = a.LT / a.Mb;
    const StepDesc sd = a.sd[s];
    const MapSnap ms = a.snap[s];
    const int nb = (sd.n + a.Mb - 1) / a.Mb, nt = (ms.NL + a.LT - 1) / a.LT;
    if (w < 0 ? c >= nb : w >= nb + (nt - 1) * hop) return;
    float2 v[16];
    if (w < 0) {
        const float nh = (float)ms.nuc, nl = (float)(ms.nuc - (double)nh);
        if (t < 16) s_step[t] = cis_df(nh, nl, (float)(T * t));
        __syncthreads();
        const float2 base = cis_df(nh, nl, (float)(c * a.Mb + t));
        const int len = min(a.Mb, sd.n - c * a.Mb);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int m = t + T * e;
            v[e] = m < len ? cmul(load_sample(sd.y1, sd.fmt, c * a.Mb + m), cmul(base, s_step[e])) : make_float2(0.f, 0.f);
        }
    } else {
        const int64_t i0 = (int64_t)w * a.Mb + ms.L0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int64_t i = i0 + t + T * e;
            v[e] = i >= 0 && i < sd.n ? load_sample(sd.y2, sd.fmt, (int)i) : make_float2(0.f, 0.f);
        }
    }
    fft_cta<LOGN>(v, sm, a.tw);
    float2 *F = a.F2 + ((size_t)s * (a.Cmax + a.nwin) + c) * n + t;
#pragma unroll
    for (int e = 0; e < 16; ++e) F[T * e] = v[e];
}

template <int LOGN>
__global__ void __launch_bounds__((1 << LOGN) / 16, LOGN == 14 ? 1 : LOGN == 13 ? 2 : 768 * 16 / (1 << LOGN)) k_chunk_corr(MapArgs a)
{
    constexpr int n = 1 << LOGN, T = n / 16;
    extern __shared__ __align__(16) float2 sm[];
    const int t = threadIdx.x, c = blockIdx.x, tile = blockIdx.y, s = blockIdx.z;
    const MapSnap ms = a.snap[s];
    if (c * a.Mb >= a.sd[s].n || tile * a.LT >= ms.NL) return;
    const float2 *Fs = a.F2 + (size_t)s * (a.Cmax + a.nwin) * n + t;
    const float2 *F1 = Fs + (size_t)c * n, *F2 = Fs + (size_t)(a.Cmax + c + tile * (a.LT / a.Mb)) * n;
    constexpr float inv = 1.0f / (float)n;
    float2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const float2 g = __ldg(F1 + T * e), f = __ldg(F2 + T * e);
        v[e] = make_float2(fmaf(g.x, f.x, g.y * f.y) * inv, fmaf(g.y, f.x, -g.x * f.y) * inv);
    }
    fft_cta<LOGN>(v, sm, a.tw);
    float2 *U = a.U + ((size_t)s * a.Cmax + c) * a.NLpad;
    const int l0 = tile * a.LT, nl_t = min(a.LT, ms.NL - l0);
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int l = t + T * e;
        if (l < nl_t) U[l0 + l] = v[e];
    }
}

// X[q][l]: a warp takes 32 lags and NQ bins (in pairs: the packed FMAs run
// over two bins, whose node weights lie side by side in shared memory); the
// CTA's warps share the lags (their U loads hit L1). Per block and node a
// warp loads 256 bytes of U and 4 NQ bytes of weights for 2 NQ x 32 FMAs.
constexpr int kExpWarps = 8;

// LW of the CTA's warps lie along the lags (32 each), 8 / LW along the bins:
// narrow tables (few bins) take more lags per CTA. U and the phases are staged
// exp_rows (block, node) rows at a time, so a stage's barrier is paid once for
// several blocks where a block has few nodes.
__host__ __device__ constexpr int exp_rows(int NQ) { return NQ >= 16 ? 96 : 48; }
template <int NQ, int LW> __global__ void __launch_bounds__(32 * kExpWarps) k_map_expand(MapArgs a)
{
    constexpr int QW = kExpWarps / LW, NB = NQ * QW, H = NQ / 2, T = 32 * kExpWarps, NLC = 32 * LW;
    extern __shared__ __align__(16) float sm_f[];
    const int s = blockIdx.z, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const StepDesc sd = a.sd[s % a.ksd];
    const MapSnap ms = a.snap[s];
    const int qb = blockIdx.y * NB, P = a.P, CS = max(1, exp_rows(NQ) / P);  // blocks per stage
    const int l0 = blockIdx.x * NLC;
    if (l0 >= ms.NL) return;
    float *sT = sm_f;                                              // [P][NB]
    float2 *sE = reinterpret_cast<float2 *>(sT + P * NB);          // [3][CS][NB]
    float2 *sU = sE + 3 * CS * NB;                                 // [3][CS P][NLC]
    const int C = (sd.n + a.Mb - 1) / a.Mb, NS = (C + CS - 1) / CS;
    const float2 *U = a.U + (size_t)s * a.Cmax * P * a.NLpad + l0;
    const float2 *E = a.phase + (size_t)s * a.Cmax * a.Q;
    const int lw = min(NLC, a.NLpad - l0);  // lags of the tile that exist in U (a multiple of 32)
    auto stage = [&](int g) {  // the U rows and phases of blocks g CS .. , asynchronously
        if (g < NS) {
            const int nc = min(CS, C - g * CS);
            float2 *u = sU + (g % 3) * CS * P * NLC;
            for (int i = threadIdx.x; i < nc * P * NLC; i += T)
                if (i % NLC < lw) cp_async8(u + i, U + ((size_t)g * CS * P + i / NLC) * a.NLpad + i % NLC);
            for (int i = threadIdx.x; i < nc * NB; i += T)
                cp_async8(sE + (g % 3) * CS * NB + i, E + (size_t)(g * CS + i / NB) * a.Q + min(qb + i % NB, a.Q - 1));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0);
    stage(1);
    for (int i = threadIdx.x; i < P * NB; i += T) {
        const int q = qb + i % NB;
        sT[i] = q < a.Q ? __ldg(a.T + (i / NB) * a.Q + q) : 0.f;
    }
    const int wq = warp % QW, wl = warp / QW, q0 = qb + NQ * wq;
    float2 xr[H], xi[H];  // real and imaginary parts of bin pairs
#pragma unroll
    for (int i = 0; i < H; ++i) xr[i] = xi[i] = make_float2(0.f, 0.f);
    for (int g = 0; g < NS; ++g) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();  // stage g in place; every warp is done with stage g - 1, whose slot takes g + 2
        stage(g + 2);
        if (q0 >= a.Q) continue;
        const int nc = min(CS, C - g * CS);
        const float2 *u_s = sU + (g % 3) * CS * P * NLC + 32 * wl + lane;
        for (int cc = 0; cc < nc; ++cc) {
            const float *t_s = sT + NQ * wq;
            float2 yr[H], yi[H];
#pragma unroll
            for (int i = 0; i < H; ++i) yr[i] = yi[i] = make_float2(0.f, 0.f);
#pragma unroll 2
            for (int p = 0; p < P; ++p) {
                const float2 u = *u_s;
                u_s += NLC;
                const float2 ur = make_float2(u.x, u.x), ui = make_float2(u.y, u.y);
#pragma unroll
                for (int i = 0; i < H; i += 2) {
                    const float4 t = *reinterpret_cast<const float4 *>(t_s + NB * p + 2 * i);
                    const float2 ta = make_float2(t.x, t.y), tb = make_float2(t.z, t.w);
                    yr[i] = fma2(ta, ur, yr[i]);
                    yi[i] = fma2(ta, ui, yi[i]);
                    yr[i + 1] = fma2(tb, ur, yr[i + 1]);
                    yi[i + 1] = fma2(tb, ui, yi[i + 1]);
                }
            }
            const float4 *e_s = reinterpret_cast<const float4 *>(sE + ((g % 3) * CS + cc) * NB + NQ * wq);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const float4 e = e_s[i];  // two bins' phases
                const float2 er = make_float2(e.x, e.z), ei = make_float2(e.y, e.w);
                xr[i] = fma2(er, yr[i], fma2(make_float2(-ei.x, -ei.y), yi[i], xr[i]));
                xi[i] = fma2(er, yi[i], fma2(ei, yr[i], xi[i]));
            }
        }
    }
    const int l = l0 + 32 * wl + lane;
    if (l >= ms.NL || q0 >= a.Q) return;
    const int L = ms.L0 + l;
    const bool none = L >= sd.n || L <= -sd.n;  // no overlap: exactly zero
#pragma unroll
    for (int i = 0; i < NQ; ++i)
        if (q0 + i < a.Q) {
            const float2 v = i & 1 ? make_float2(xr[i / 2].y, xi[i / 2].y) : make_float2(xr[i / 2].x, xi[i / 2].x);
            a.X[((size_t)s * a.Q + q0 + i) * a.NLpad + l] = none ? make_float2(0.f, 0.f) : v;
        }
}

// Whether lag L's overlap touches a sample that is not finite: n runs over
// [max(0, -L), min(N, N - L)), y2's index over [max(0, L), min(N, N + L)).
__device__ __forceinline__ bool lag_bad(int4 b, int L, int N)
{
    if (L >= N || L <= -N) return false;
    return L >= 0 ? (b.x < N - L || b.w >= L) : (b.y >= -L || b.z < N + L);
}

// Nearest integer of |x| < 2^22, as a float and as an integer, by the
// round-off of 1.5 x 2^23 (two additions on the FP32 pipe where the
// conversion instructions run at a fraction of its rate).
__device__ __forceinline__ float round_magic(float x, int &n)
{
    constexpr float magic = 12582912.f;
    const float y = __fadd_rn(x, magic);
    n = __float_as_int(y) - 0x4b400000;
    return __fsub_rn(y, magic);
}

// The 6-point Lagrange weights of nodes at -2.5, -1.5, ..., 2.5 at s in
// [-0.5, 0.5]: the pair +-n has E(s^2) (1 +- s / n), E the quadratic through
// the other nodes' squares; E and E / n as one packed polynomial.
__device__ __forceinline__ void weights6(float s, float (&w)[6])
{
    const float s2 = s * s;
    const float2 q = make_float2(s2, s2);
    auto pair = [&](float d, float inv_n, float b, float c) {
        const float2 k2 = make_float2(d, d * inv_n), k1 = make_float2(d * b, d * b * inv_n),
                     k0 = make_float2(d * c, d * c * inv_n);
        return fma2(fma2(k2, q, k1), q, k0);
    };
    const float2 a = pair(1.f / 24.f, 2.f, -8.5f, 14.0625f);
    const float2 b = pair(-1.f / 16.f, 1.f / 1.5f, -6.5f, 1.5625f);
    const float2 c = pair(1.f / 48.f, 0.4f, -2.5f, 0.5625f);
    w[0] = fmaf(-s, c.y, c.x);
    w[1] = fmaf(-s, b.y, b.x);
    w[2] = fmaf(-s, a.y, a.x);
    w[3] = fmaf(s, a.y, a.x);
    w[4] = fmaf(s, b.y, b.x);
    w[5] = fmaf(s, c.y, c.x);
}

// Whether a table of NL lags and Q bins holds lag l (from its first) and the six bins
// around bin coordinate U0 + u (Lagrange4 reads the lags l - 1 .. l + 2).
template <bool FRAC> __device__ __forceinline__ bool in_table(int l, int NL, int U0, float u, int Q)
{
    int k;
    round_magic(u - 0.5f, k);
    return (unsigned)(FRAC ? l - 1 : l) < (unsigned)(FRAC ? NL - 3 : NL) && (unsigned)(U0 + k - 2) <= (unsigned)(Q - 6);
}

// One candidate and snapshot, at bin coordinate U0 + u: |C|^2 or |C|. BAD:
// some capture may hold samples that are not finite. The host's bounds keep
// lag and bins inside the table, which the callers check (in_table: a node outside
// reports itself, as to the lag sort of the contraction); an index that falls
// outside of its memory reads its start.
template <bool FRAC, bool BAD>
__device__ __forceinline__ float map_value(const MapArgs &a, const float2 *__restrict__ X, int s, int L0, int L,
                                           float mu, int U0, float u)
{
    // bins q0 - 2 .. q0 + 3, q0 <= U0 + u <= q0 + 1, at its middle plus t
    int k;
    const float t = (u - 0.5f) - round_magic(u - 0.5f, k);
    float w[6];
    weights6(t, w);
    int idx = (U0 + k - 2) * a.NLpad + (L - L0);
    if (FRAC) {
        if ((unsigned)(idx - 1) > (unsigned)((a.Q - 5) * a.NLpad - 4)) idx = 1;
    } else {
        if ((unsigned)idx >= (unsigned)((a.Q - 5) * a.NLpad)) idx = 0;
    }
    const float2 *R = X + idx;
    float cx = 0.f, cy = 0.f;
    if (!FRAC) {
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            const float2 v = __ldg(R + (size_t)e * a.NLpad);
            cx = fmaf(w[e], v.x, cx);
            cy = fmaf(w[e], v.y, cy);
        }
    } else {
        const float lw[4] = {-mu * (mu - 1.f) * (mu - 2.f) * (1.f / 6.f), (mu + 1.f) * (mu - 1.f) * (mu - 2.f) * 0.5f,
                             -(mu + 1.f) * mu * (mu - 2.f) * 0.5f, (mu + 1.f) * mu * (mu - 1.f) * (1.f / 6.f)};
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            float zx = 0.f, zy = 0.f;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float2 v = __ldg(R + (size_t)e * a.NLpad + m - 1);
                zx = fmaf(lw[m], v.x, zx);
                zy = fmaf(lw[m], v.y, zy);
            }
            cx = fmaf(w[e], zx, cx);
            cy = fmaf(w[e], zy, cy);
        }
    }
    if (BAD) {
        const int4 b = __ldg(reinterpret_cast<const int4 *>(a.bad) + s);
        const int N = a.sd[s].n;
        bool bad = lag_bad(b, L, N);
        if (FRAC) bad |= lag_bad(b, L - 1, N) || lag_bad(b, L + 1, N) || lag_bad(b, L + 2, N);
        if (bad) return __int_as_float(0x7fc00000);
    }
    const float pw = fmaf(cx, cx, cy * cy);
    return a.acc == DG_ACC_POWER ? pw : sqrtf(pw);
}

// Lag, fractional delay and bin coordinate U0 + u of one node in one snapshot, from
// the double-float geometry (the lag by the FP64 expression where D lies
// within 1e-6 of a rounding boundary); false when |D| is out of range. The
// coordinate is formed in double-float: with one FP32 product the surface of a table
// of 4000 bins was off by 1.7e-5, now 7e-7.
template <bool FRAC>
__device__ __forceinline__ bool map_node(const MapArgs &a, const MapSnap &ms, int s, const double *node, const dfl (&xyz)[3],
                                         int &L, float &mu, int &U0, float &u)
{
    dfl ed[12], D, nu;
#pragma unroll
    for (int t = 0; t < 12; ++t) ed[t] = {__ldg(a.ephf + 24 * (size_t)s + 2 * t), __ldg(a.ephf + 24 * (size_t)s + 2 * t + 1)};
    geometry_dfl(xyz[0], xyz[1], xyz[2], ed, {a.fsc_hi, a.fsc_lo}, {a.ilf_hi, a.ilf_lo}, D, nu);
    const dfl df = df_two_sum(nu.hi, -ms.nu0_hi);
    const float p = df.hi * ms.inv_delta;
    const float tail = fmaf(df.hi, ms.inv_delta_lo, fmaf(df.lo + (nu.lo - ms.nu0_lo), ms.inv_delta, fmaf(df.hi, ms.inv_delta, -p)));
    u = (p - round_magic(p, U0)) + tail;
    mu = 0.f;
    if (!(fabsf(D.hi) < 1.0e9f)) return false;
    if (FRAC ? floor_df(D, L, mu) : round_df(D, L)) return true;
    double e[12], D64, nu64;
    for (int t = 0; t < 12; ++t) e[t] = a.eph[12 * (size_t)s + t];
    geometry(node[0], node[a.G], node[2 * a.G], e, a.fs, a.lambda, D64, nu64);
    if (!(fabs(D64) < 1.0e9)) return false;
    L = lag_of(D64, FRAC ? DG_DELAY_LAGRANGE4 : DG_DELAY_INTEGER);
    mu = (float)(D64 - (double)L);
    return true;
}

// Polynomial geometry. On a tile whose radius h is small against the range
// rho to the receivers, D and the FDOA are smooth: the m-th Taylor term of
// D is at most m |p2 - p1| fs / c (h / rho)^m. A warp evaluates the
// double-float geometry at kPolyPts nodes of the tile (a 6 x 6 Chebyshev-like
// lattice without its corners) and fits polynomials of total degree 5 in the
// normalised offsets by a constant least-squares matrix; the host takes a
// tile only where the bound on the truncation stays below 2e-6 samples.
// Precision: D = I0 + gu r + gv c + P(r, c) with an integer I0 and slopes
// that are multiples of 2^-13, so the linear part is exact in FP32 at every
// node (|offset| <= 31.5, |slope| < 8: 23 bits), and only P, a few samples at
// most, is rounded (about 5e-7).
__device__ __forceinline__ float2 poly_offset(const MapArgs &a, int r, int c)  // from the tile's centre
{
    return make_float2((float)r - 0.5f * (float)(a.poly.rows - 1), (float)c - 0.5f * (float)(kPolyCols - 1));
}

constexpr int kPolyWarps = 8;
static_assert(4 + 2 * kPolyTerms + 2 <= kPolyStride, "the flag lies behind the terms");
__global__ void __launch_bounds__(32 * kPolyWarps) k_map_poly(MapArgs a, int tiles_j, int64_t pairs)
{
    __shared__ float s_fit[kPolyTerms][kPolyPts + 1];
    __shared__ float2 s_val[kPolyWarps][kPolyPts];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kPolyTerms * kPolyPts; i += 32 * kPolyWarps)
        s_fit[i / kPolyPts][i % kPolyPts] = __ldg(a.fit + i);
    __syncthreads();
    const int64_t w = blockIdx.x * (int64_t)kPolyWarps + warp;
    if (w >= pairs) return;
    const int s = (int)(w % a.S);
    const int64_t tile = w / a.S;
    const int r0 = min((int)(tile / tiles_j) * a.poly.rows, a.nrows - a.poly.rows);
    const int c0 = min((int)(tile % tiles_j) * kPolyCols, a.nlon - kPolyCols);
    const MapSnap ms = a.snap[s];
    const int pr = a.poly.pr[lane], pc = a.poly.pc[lane];
    const int64_t p = (int64_t)(r0 + pr) * a.nlon + c0 + pc;
    dfl ed[12], D, nu;
#pragma unroll
    for (int t = 0; t < 12; ++t) ed[t] = {__ldg(a.ephf + 24 * (size_t)s + 2 * t), __ldg(a.ephf + 24 * (size_t)s + 2 * t + 1)};
    geometry_dfl(df_from(a.xyz[p]), df_from(a.xyz[a.G + p]), df_from(a.xyz[2 * a.G + p]), ed, {a.fsc_hi, a.fsc_lo},
                 {a.ilf_hi, a.ilf_lo}, D, nu);
    constexpr unsigned all = 0xffffffffu;
    constexpr int mid = 18;  // a sample near the centre anchors both
    float I0 = rintf(__shfl_sync(all, D.hi, mid));
    const dfl nr = {__shfl_sync(all, nu.hi, mid), __shfl_sync(all, nu.lo, mid)};
    const dfl ur = df_mul(df_sub(nr, {ms.nu0_hi, ms.nu0_lo}), {ms.inv_delta, ms.inv_delta_lo});
    const float U0 = rintf(ur.hi);
    const float du = ((nu.hi - nr.hi) + (nu.lo - nr.lo)) * ms.inv_delta + ((ur.hi - U0) + ur.lo);
    const float dD = (D.hi - I0) + D.lo;
    // slopes per node from the linear terms (c^1: term 1, r^1: term 6)
    const float hr = 0.5f * (float)(a.poly.rows - 1), hc = 0.5f * (float)(kPolyCols - 1);
    float g0 = s_fit[0][lane] * dD, gc = s_fit[1][lane] * dD, gr = s_fit[6][lane] * dD;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        g0 += __shfl_xor_sync(all, g0, d);
        gc += __shfl_xor_sync(all, gc, d);
        gr += __shfl_xor_sync(all, gr, d);
    }
    I0 += rintf(g0);  // the centre's
    gr = rintf(gr / hr * 8192.f) * (1.f / 8192.f);
    gc = rintf(gc / hc * 8192.f) * (1.f / 8192.f);
    const float2 o = poly_offset(a, pr, pc);
    // D.hi - I0 and the linear part are multiples of 2^-14 or finer parts of D.hi: exact difference
    s_val[warp][lane] = make_float2(((D.hi - I0) - fmaf(gr, o.x, gc * o.y)) + D.lo, du);
    __syncwarp();
    float *out = a.coef + (size_t)w * kPolyStride;
    float2 c = make_float2(0.f, 0.f);
    if (lane < kPolyTerms) {
#pragma unroll 8
        for (int i = 0; i < kPolyPts; ++i) {
            const float2 v = s_val[warp][i];
            c.x = fmaf(s_fit[lane][i], v.x, c.x);
            c.y = fmaf(s_fit[lane][i], v.y, c.y);
        }
        *reinterpret_cast<float2 *>(out + 4 + 2 * lane) = c;
    } else if (lane == kPolyTerms) {
        *reinterpret_cast<float4 *>(out) = make_float4(I0, U0, gr, gc);
    }
    // D and the bin coordinate over the tile: the constant terms and the sums of the
    // others' magnitudes (the offsets are at most 1). 1 behind the terms where
    // that does not put every node of the tile inside the table: the lookup then checks
    // each (checking all of them there cost 7 % of the large lookup).
    const float2 mid0 = make_float2(__shfl_sync(all, c.x, 0), __shfl_sync(all, c.y, 0));
    float rd = lane ? fabsf(c.x) : fabsf(gr) * hr + fabsf(gc) * hc, ru = lane ? fabsf(c.y) : 0.f;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        rd += __shfl_xor_sync(all, rd, d);
        ru += __shfl_xor_sync(all, ru, d);
    }
    if (lane == kPolyTerms + 1) {
        const bool frac = a.delay != DG_DELAY_INTEGER;
        const float dm = (I0 - (float)ms.L0) + mid0.x, um = U0 + mid0.y;
        const float m = frac ? 1.01f : 0.51f, p = frac ? 2.01f : 0.51f;
        const bool in = dm - rd > m && dm + rd < (float)(ms.NL - 1) - p && um - ru > 2.01f && um + ru < (float)a.Q - 3.01f;
        *reinterpret_cast<float2 *>(out + 4 + 2 * kPolyTerms) = make_float2(in ? 0.f : 1.f, 0.f);
    }
}

// The lookup of a tile of poly.rows x 32 nodes by one CTA: a warp takes a
// compact 4-row x 8-column patch per step (their lags, and so their table
// addresses, lie close together), R = rows / 8 steps of 4 rows; a thread's
// column is fixed, so the polynomials collapse to one variable per snapshot.
template <bool FRAC, bool BAD, int R>
__global__ void __launch_bounds__(256, 4) k_map_lookup_poly(MapArgs a, int tiles_j)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x, ti = tile / tiles_j, tj = tile % tiles_j;
    constexpr int TR = 8 * R;
    const int r0 = min(ti * TR, a.nrows - TR), c0 = min(tj * kPolyCols, a.nlon - kPolyCols);
    const int j = tj * kPolyCols + (warp & 3) * 8 + (lane & 7);
    const int i0 = ti * TR + (warp >> 2) * (4 * R) + (lane >> 3);
    const float2 o = poly_offset(a, i0 - r0, j - c0);
    const float vn = o.y * (2.f / (float)(kPolyCols - 1));
    float sum[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = i0 + 4 * r;
        sum[r] = (!a.first && i < a.nrows && j < a.nlon) ? a.out[(int64_t)i * a.nlon + j] : 0.f;
    }
    const float4 *cf = reinterpret_cast<const float4 *>(a.coef + (size_t)tile * a.S * kPolyStride);
    const float2 vn2 = make_float2(vn, vn);
    const float2 *X = a.X;
    for (int s = 0; s < a.S; ++s, cf += kPolyStride / 4, X += (size_t)a.Q * a.NLpad) {
        const int L0 = a.snap[s].L0;
        const float4 head = __ldg(cf);
        // polynomials in the row offset: x D, y bin coordinate; terms of
        // r^0 (c^0..5), r^1 (c^0..4), r^2 (c^0..3), ...
        float2 cr[6];
        bool check;
        {
            float2 m[22];
#pragma unroll
            for (int t = 0; t < 11; ++t) {
                const float4 f = __ldg(cf + 1 + t);
                m[2 * t] = make_float2(f.x, f.y);
                m[2 * t + 1] = make_float2(f.z, f.w);
            }
            int at = 0;
#pragma unroll
            for (int e = 0; e < 6; ++e) {
                float2 h = m[at + 5 - e];
#pragma unroll
                for (int b = 4 - e; b >= 0; --b) h = fma2(h, vn2, m[at + b]);
                cr[e] = h;
                at += 6 - e;
            }
            check = m[21].x != 0.f;  // k_map_poly: some node of the tile may lie outside the table
        }
        const float lin_c = head.w * o.y;
        const int I0 = (int)head.x, U0 = (int)head.y;
        if (check) {
            const int NL = a.snap[s].NL;
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const float rr = o.x + 4.f * r, un = rr * (2.f / (float)(TR - 1));
                const float2 un2 = make_float2(un, un);
                float2 h = cr[5];
#pragma unroll
                for (int e = 4; e >= 0; --e) h = fma2(h, un2, cr[e]);
                const float lin = fmaf(head.z, rr, lin_c);
                int n1, n2;
                const float t = (lin - round_magic(lin, n1)) + h.x;
                round_magic(FRAC ? t - 0.5f : t, n2);
                // an integer lag next to its rounding boundary may be the next one
                if (i0 + 4 * r < a.nrows && j < a.nlon && !in_table<FRAC>(I0 + n1 + n2 - L0, NL, U0, h.y, a.Q))
                    atomicOr(a.err, ERR_LAG_RANGE);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float rr = o.x + 4.f * r;
            const float un = rr * (2.f / (float)(TR - 1));
            const float2 un2 = make_float2(un, un);
            float2 h = cr[5];
#pragma unroll
            for (int e = 4; e >= 0; --e) h = fma2(h, un2, cr[e]);
            const float lin = fmaf(head.z, rr, lin_c);  // exact
            int n1, n2;
            const float t = (lin - round_magic(lin, n1)) + h.x;  // D = I0 + n1 + t
            const float mu = t - round_magic(FRAC ? t - 0.5f : t, n2);
            int L = I0 + n1 + n2;  // Lagrange4: floor, or one less with mu = 1 at an integer
            if (!FRAC && fabsf(mu) > 0.5f - 1e-5f) {  // within 1e-5 of a rounding boundary: the FP64 expression
                const int i = min(i0 + 4 * r, a.nrows - 1);
                double e[12], D64, nu64;
                for (int q = 0; q < 12; ++q) e[q] = a.eph[12 * (size_t)s + q];
                const int64_t p = (int64_t)i * a.nlon + min(j, a.nlon - 1);
                geometry(a.xyz[p], a.xyz[a.G + p], a.xyz[2 * a.G + p], e, a.fs, a.lambda, D64, nu64);
                L = lag_of(D64, DG_DELAY_INTEGER);
            }
            const float v = map_value<FRAC, BAD>(a, X, s, L0, L, mu, U0, h.y);
            sum[r] = (s == 0 && a.first) ? v : sum[r] + v;
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = i0 + 4 * r;
        if (i < a.nrows && j < a.nlon) a.out[(int64_t)i * a.nlon + j] = sum[r];
    }
}

// One thread per node (32 consecutive nodes of a grid row per warp); WK warps
// of a CTA share the nodes and split the snapshots, 8 / WK take their own
// rows. WK = 8 serves small grids, which would leave the chip idle otherwise:
// the partial values meet in shared memory and are added in snapshot order.
template <bool FRAC, bool BAD, int WK> __global__ void __launch_bounds__(256) k_map_lookup(MapArgs a)
{
    constexpr int WN = 8 / WK;
    __shared__ float s_val[WK > 1 ? WK : 1][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles_j = (a.nlon + 31) / 32, reg = blockIdx.y;
    const double *xyz_r = a.xyz + 3 * a.G * reg;
    float *out = a.out + a.G * reg;
    const float2 *X = a.X + (size_t)reg * a.ksd * a.Q * a.NLpad;
    const MapSnap *snap = a.snap + (size_t)reg * a.ksd;
    const int tj = blockIdx.x % tiles_j, ti = blockIdx.x / tiles_j;
    const int i = ti * WN + (WK > 1 ? warp / WK : warp), j = tj * 32 + lane;
    const int wk = WK > 1 ? warp % WK : 0;
    const bool ok = i < a.nrows && j < a.nlon;
    const int64_t p = (int64_t)min(i, a.nrows - 1) * a.nlon + min(j, a.nlon - 1);
    dfl xyz[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) xyz[d] = df_from(xyz_r[d * a.G + p]);
    float sum = a.first ? 0.f : out[p];
    bool any = !a.first;
    for (int k = 0; k < a.ksd; k += WK) {
        const int s = k + wk;
        float v = 0.f;
        if (s < a.ksd) {
            const MapSnap ms = snap[s];
            int L, U0;
            float mu, u;
            if (map_node<FRAC>(a, ms, s, xyz_r + p, xyz, L, mu, U0, u)) {
                if (!in_table<FRAC>(L - ms.L0, ms.NL, U0, u, a.Q) && ok) atomicOr(a.err, ERR_LAG_RANGE);
                v = map_value<FRAC, BAD>(a, X + (size_t)s * a.Q * a.NLpad, s, ms.L0, L, mu, U0, u);
            } else if (ok) {
                atomicOr(a.err, ERR_LAG_RANGE);
            }
        }
        if (WK == 1) {
            sum = any ? sum + v : v;
            any = true;
        } else {
            s_val[wk][lane] = v;
            __syncthreads();
            if (wk == 0)
                for (int w = 0; w < WK && k + w < a.ksd; ++w) {
                    sum = any ? sum + s_val[w][lane] : s_val[w][lane];
                    any = true;
                }
            __syncthreads();
        }
    }
    if (ok && wk == 0) out[p] = sum;
}

// Tables of a grid of a few lags (the refinement around a node). Its band is
// so narrow that the phase turns by a fraction of a cycle over a capture:
// with nu_c the centre's FDOA and t = (n - N/2) tscale in [-1, 1],
//     X(l, nu) = sum_m j^m c_m(nu) S[m][l],
//     S[m][l] = sum_n y1[n] e^{j 2 pi nu_c (n - N/2)} conj(y2[n + l]) T_m(t),
// the Chebyshev series of e^{j 2 pi (nu - nu_c)(n - N/2)} cut after P terms (real
// weights: 2 FMAs per term where a turned copy of y1 per Doppler node takes
// 4 and a shared load). A CTA walks blocks of samples of one snapshot: y1
// turned to nu_c and the window of y2 in shared memory; a warp takes 4 lags of
// a share of the samples (5 shared loads for 16 + 8 P FMAs). The CTAs' sums are
// added in a fixed order by k_map_few_x, which also expands the terms to the
// table's bins.
constexpr int kFewLags = 4;  // lags per warp

// v[i] summed over the warp's lanes: halves are exchanged while the count is
// even, so each lane ends with N / 32 of the sums (or a pair of lanes with
// the same 3 for N = 48); returns this lane's first index.
template <int N> __device__ __forceinline__ int warp_scatter_sum(float *v, int lane)
{
    int first = 0, n = N;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        if (n % 2 == 0) {
            n /= 2;
            const bool up = lane & d;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                if (i >= n) break;
                const float send = up ? v[i] : v[i + n];
                const float keep = up ? v[i + n] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
            }
            if (up) first += n;
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (i >= n) break;
                v[i] += __shfl_xor_sync(0xffffffffu, v[i], d);
            }
        }
    }
    return first;
}

template <int P> __global__ void __launch_bounds__(256) k_map_few(MapArgs a, MapFew f)
{
    constexpr int NV = 2 * kFewLags * P;  // floats per lag group
    __shared__ __align__(16) float2 y1t[kFewBlock], y2w[kFewBlock + kFewMaxLags];
    __shared__ float s_red[8][NV];
    __shared__ float s_nu[2];
    __shared__ int s_L0;
    const int s = blockIdx.y, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const StepDesc sd = a.sd[s];
    const int N = sd.n;
    if (t == 0) {  // the centre's geometry
        dfl ed[12], D, nu;
        for (int q = 0; q < 12; ++q) ed[q] = {__ldg(a.ephf + 24 * (size_t)s + 2 * q), __ldg(a.ephf + 24 * (size_t)s + 2 * q + 1)};
        geometry_dfl(df_from(a.xyz[f.centre]), df_from(a.xyz[a.G + f.centre]), df_from(a.xyz[2 * a.G + f.centre]), ed,
                     {a.fsc_hi, a.fsc_lo}, {a.ilf_hi, a.ilf_lo}, D, nu);
        const int L0 = (int)floor((double)D.hi + (double)D.lo - f.md - 0.51) - (a.delay != DG_DELAY_INTEGER ? 1 : 0);
        s_L0 = L0;
        s_nu[0] = nu.hi;
        s_nu[1] = nu.lo;
        if (blockIdx.x == 0) {
            MapSnap ms;
            ms.nuc = (double)nu.hi + (double)nu.lo;
            ms.nu0 = ms.nuc - f.halfw;
            ms.delta = f.delta;
            ms.halfw = f.halfw;
            ms.nu0_hi = (float)ms.nu0;
            ms.nu0_lo = (float)(ms.nu0 - (double)ms.nu0_hi);
            ms.inv_delta = (float)(1.0 / f.delta);
            ms.inv_delta_lo = (float)(1.0 / f.delta - (double)ms.inv_delta);
            ms.L0 = L0;
            ms.NL = a.LT;
            f.snap[s] = ms;
        }
    }
    __syncthreads();
    const int L0 = s_L0, NG = (a.LT + kFewLags - 1) / kFewLags;
    const float nh = s_nu[0], nl = s_nu[1];
    const int NS = 8 / NG, g = warp % NG, sg = warp / NG;  // lag group, share of the samples
    float v[NV];  // [lag][term][re, im]
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.f;
    for (int64_t n0 = (int64_t)blockIdx.x * kFewBlock; n0 < N; n0 += (int64_t)gridDim.x * kFewBlock) {
        __syncthreads();
        for (int i = t; i < kFewBlock + kFewLags * NG; i += 256) {
            const int64_t q = n0 + L0 + i;
            y2w[i] = q >= 0 && q < N ? load_sample(sd.y2, sd.fmt, (int)q) : make_float2(0.f, 0.f);
        }
        for (int i = t; i < kFewBlock; i += 256) {
            const int64_t n = n0 + i;
            const float2 y = n < N ? load_sample(sd.y1, sd.fmt, (int)n) : make_float2(0.f, 0.f);
            y1t[i] = cmul(y, cis_df(nh, nl, (float)((int)n - N / 2)));
        }
        __syncthreads();
        if (sg < NS) {
            const float2 *b = y2w + kFewLags * g;
            const float t0 = (float)((int)n0 - N / 2) * f.tscale;
            for (int m = 32 * sg + lane; m < kFewBlock; m += 32 * NS) {
                const float2 y = y1t[m];
                const float x = fmaf((float)m, f.tscale, t0), x2 = 2.f * x;
#pragma unroll
                for (int l = 0; l < kFewLags; ++l) {
                    const float2 w = b[m + l];
                    const float zx = fmaf(y.x, w.x, y.y * w.y), zy = fmaf(y.y, w.x, -y.x * w.y);
                    float *o = v + 2 * l * P;
                    float tp = 1.f, tq = x;  // T_{m}, T_{m + 1}
                    o[0] += zx;
                    o[1] += zy;
#pragma unroll
                    for (int p = 1; p < P; ++p) {
                        o[2 * p] = fmaf(tq, zx, o[2 * p]);
                        o[2 * p + 1] = fmaf(tq, zy, o[2 * p + 1]);
                        const float tn = fmaf(x2, tq, -tp);
                        tp = tq;
                        tq = tn;
                    }
                }
            }
        }
    }
    if (sg < NS) {
        const int first = warp_scatter_sum<NV>(v, lane);
        constexpr int per = NV % 32 == 0 ? NV / 32 : NV / 16;
#pragma unroll
        for (int i = 0; i < per; ++i) s_red[warp][first + i] = v[i];
    }
    __syncthreads();
    float *out = reinterpret_cast<float *>(a.U) + ((size_t)s * a.Cmax + blockIdx.x) * (size_t)(NG * NV);
    for (int i = t; i < NG * NV; i += 256) {
        float x = 0.f;
        for (int w = 0; w < NS; ++w) x += s_red[i / NV + w * NG][i % NV];
        out[i] = x;
    }
}

template <int P> __global__ void __launch_bounds__(256) k_map_few_x(MapArgs a, MapFew f)
{
    constexpr int NV = 2 * kFewLags * P;
    __shared__ float s_sum[kFewMaxLags / kFewLags * NV];
    const int s = blockIdx.x, t = threadIdx.x;
    const int N = a.sd[s].n, n = (a.LT + kFewLags - 1) / kFewLags * NV;
    const float *U = reinterpret_cast<const float *>(a.U) + (size_t)s * a.Cmax * n;
    for (int i = t; i < n; i += 256) {
        float x = 0.f;
#pragma unroll 8
        for (int c = 0; c < a.Cmax; ++c) x += __ldg(U + (size_t)c * n + i);
        s_sum[i] = x;
    }
    __syncthreads();
    const int L0 = f.snap[s].L0;
    for (int i = t; i < a.Q * a.LT; i += 256) {
        const int q = i / a.LT, l = i % a.LT, L = L0 + l;
        float2 x = make_float2(0.f, 0.f);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float *v = s_sum + (l / kFewLags) * NV + 2 * ((l % kFewLags) * P + p);
            const float c = f.T[p * a.Q + q];
            if (p % 4 == 0) {  // times j^p
                x.x = fmaf(c, v[0], x.x);
                x.y = fmaf(c, v[1], x.y);
            } else if (p % 4 == 1) {
                x.x = fmaf(-c, v[1], x.x);
                x.y = fmaf(c, v[0], x.y);
            } else if (p % 4 == 2) {
                x.x = fmaf(-c, v[0], x.x);
                x.y = fmaf(-c, v[1], x.y);
            } else {
                x.x = fmaf(c, v[1], x.x);
                x.y = fmaf(-c, v[0], x.y);
            }
        }
        if (L >= N || L <= -N) x = make_float2(0.f, 0.f);
        a.X[((size_t)s * a.Q + q) * a.NLpad + l] = x;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <int LOGN> static cudaError_t launch_tables(const MapArgs &a, cudaStream_t st)
{
    constexpr int n = 1 << LOGN;
    const size_t smem = sizeof(float2) * (size_t)(n + n / 16);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_map_spec<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_map_corr<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    const dim3 gs((unsigned)a.Cmax, (unsigned)a.ntile, (unsigned)a.S);
    k_map_spec<LOGN><<<gs, n / 16, smem, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const dim3 gc((unsigned)(a.Cmax * a.P), (unsigned)a.ntile, (unsigned)a.S);
    k_map_corr<LOGN><<<gc, n / 16, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_map_twiddles(float2 *tw, int logn, cudaStream_t st)
{
    const int n = 1 << logn;
    k_map_twiddles<<<(n + 255) / 256, 256, 0, st>>>(tw, n);
    return cudaGetLastError();
}

static cudaError_t launch_bad(const MapArgs &a, cudaStream_t st, int *launches)
{
    if (!a.bad) return cudaSuccess;
    k_map_bad_init<<<1, 256, 0, st>>>(a.bad, a.ksd);
    k_map_bad<<<dim3(16, (unsigned)a.ksd, 2), 256, 0, st>>>(a);
    *launches += 2;
    return cudaGetLastError();
}

size_t map_few_partials(int P, int NL) { return (size_t)((NL + kFewLags - 1) / kFewLags) * 2 * kFewLags * P; }

template <int P> static cudaError_t launch_few(const MapArgs &a, const MapFew &f, cudaStream_t st)
{
    k_map_few<P><<<dim3((unsigned)a.Cmax, (unsigned)a.S), 256, 0, st>>>(a, f);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_map_few_x<P><<<(unsigned)a.S, 256, 0, st>>>(a, f);
    return cudaGetLastError();
}

cudaError_t launch_map_few(const MapArgs &a, const MapFew &f, cudaStream_t st, int *launches)
{
    const cudaError_t e = launch_bad(a, st, launches);
    if (e != cudaSuccess) return e;
    *launches += 2;
    switch (a.P) {
    case 4: return launch_few<4>(a, f, st);
    case 6: return launch_few<6>(a, f, st);
    case 8: return launch_few<8>(a, f, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_map_tables(const MapArgs &a, cudaStream_t st, int *launches)
{
    cudaError_t e = launch_bad(a, st, launches);
    if (e != cudaSuccess) return e;
    switch (a.logn) {
    case 10: e = launch_tables<10>(a, st); break;
    case 11: e = launch_tables<11>(a, st); break;
    case 12: e = launch_tables<12>(a, st); break;
    case 13: e = launch_tables<13>(a, st); break;
    case 14: e = launch_tables<14>(a, st); break;
    default: return cudaErrorInvalidValue;
    }
    *launches += 2;
    return e;
}

template <int LOGN> static cudaError_t launch_chunks(const MapArgs &a, cudaStream_t st)
{
    constexpr int n = 1 << LOGN;
    const size_t smem = sizeof(float2) * (size_t)(n + n / 16);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_chunk_spec<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_chunk_corr<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    k_chunk_spec<LOGN><<<dim3((unsigned)(a.Cmax + a.nwin), (unsigned)a.S), n / 16, smem, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_chunk_corr<LOGN><<<dim3((unsigned)a.Cmax, (unsigned)a.ntile, (unsigned)a.S), n / 16, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_chunk_sums(const MapArgs &a, cudaStream_t st, int *launches)
{
    cudaError_t e = launch_bad(a, st, launches);
    if (e != cudaSuccess) return e;
    *launches += 2;
    switch (a.logn) {
    case 10: return launch_chunks<10>(a, st);
    case 11: return launch_chunks<11>(a, st);
    case 12: return launch_chunks<12>(a, st);
    case 13: return launch_chunks<13>(a, st);
    case 14: return launch_chunks<14>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int NQ, int LW> static cudaError_t launch_expand(const MapArgs &a, cudaStream_t st)
{
    constexpr int NB = NQ * kExpWarps / LW, NLC = 32 * LW;
    const int CS = a.P < exp_rows(NQ) ? exp_rows(NQ) / a.P : 1;
    const size_t smem = sizeof(float) * (size_t)a.P * NB + sizeof(float2) * 3 * (size_t)CS * (NB + a.P * NLC);
    const cudaError_t e = cudaFuncSetAttribute(k_map_expand<NQ, LW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 ge((unsigned)((a.NLpad + NLC - 1) / NLC), (unsigned)((a.Q + NB - 1) / NB), (unsigned)a.S);
    k_map_expand<NQ, LW><<<ge, 32 * kExpWarps, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_map_expand(const MapArgs &a, cudaStream_t st)
{
    // 16 bins per warp where the table is wide enough to fill the chip, 8 otherwise
    if (a.Q >= 128) return launch_expand<16, 1>(a, st);
    if (a.Q > 32) return launch_expand<8, 1>(a, st);
    return a.Q > 16 ? launch_expand<4, 1>(a, st) : launch_expand<4, 2>(a, st);
}

cudaError_t launch_map_poly(const MapArgs &a, cudaStream_t st)
{
    const int64_t tiles_j = (a.nlon + kPolyCols - 1) / kPolyCols;
    const int64_t pairs = tiles_j * ((a.nrows + a.poly.rows - 1) / a.poly.rows) * a.S;
    const int64_t blocks = (pairs + kPolyWarps - 1) / kPolyWarps;
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    k_map_poly<<<(unsigned)blocks, 32 * kPolyWarps, 0, st>>>(a, (int)tiles_j, pairs);
    return cudaGetLastError();
}

template <bool FRAC, bool BAD> static cudaError_t launch_lookup(const MapArgs &a, cudaStream_t st)
{
    const int64_t tiles_j = (a.nlon + 31) / 32;
    // under about four CTAs per SM of one-row warps, the warps split the snapshots
    const bool split = !a.poly.rows && tiles_j * ((a.nrows + 7) / 8) * a.nreg < 152 * 4;
    const int rows = a.poly.rows ? a.poly.rows : split ? 1 : 8;  // of a CTA
    const int64_t blocks = tiles_j * ((a.nrows + rows - 1) / rows);
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    const unsigned g = (unsigned)blocks;
    if (a.poly.rows == 64) k_map_lookup_poly<FRAC, BAD, 8><<<g, 256, 0, st>>>(a, (int)tiles_j);
    else if (a.poly.rows) k_map_lookup_poly<FRAC, BAD, 4><<<g, 256, 0, st>>>(a, (int)tiles_j);
    else if (split) k_map_lookup<FRAC, BAD, 8><<<dim3(g, (unsigned)a.nreg), 256, 0, st>>>(a);
    else k_map_lookup<FRAC, BAD, 1><<<dim3(g, (unsigned)a.nreg), 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_map_lookup(const MapArgs &a, cudaStream_t st)
{
    if (a.delay == DG_DELAY_INTEGER) return a.bad ? launch_lookup<false, true>(a, st) : launch_lookup<false, false>(a, st);
    return a.bad ? launch_lookup<true, true>(a, st) : launch_lookup<true, false>(a, st);
}

}  // namespace dg
