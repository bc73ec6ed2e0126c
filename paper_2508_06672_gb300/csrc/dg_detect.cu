// dg_detect.cu -- threshold detection of emitters on an accumulated surface
// (Algorithm 1, last step). A node is a peak when its value is >= the
// threshold and it is the maximum of the (2r+1) x (2r+1) window around it;
// among equal values the lowest linear index wins (one peak per plateau).
// Peaks are sorted by value (descending), ties by index, in one CTA.
#include <cfloat>

#include "dg_internal.cuh"

namespace dg {

// A node that its eight neighbours do not rule out (few are left) has its window
// searched by the whole warp, two to four rows at a time: a lane on its own walks (2r +
// 1)^2 dependent loads while the others wait (512^2 nodes, r = 7: 50 -> 15 us).
template <typename T>
__global__ void __launch_bounds__(256) k_detect_mark(const T *__restrict__ v, int nrows, int nlon, double thr, int r,
                                                     int cap, int *count, int64_t *cand)
{
    const int64_t G = (int64_t)nrows * nlon;
    const int lane = threadIdx.x & 31;
    for (int64_t p0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; p0 < G;
         p0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = p0 + lane;
        const bool in = p < G;
        const T x = in ? v[p] : (T)0;
        const int i = in ? (int)(p / nlon) : 0, j = in ? (int)(p % nlon) : 0;
        bool peak = in && (double)x >= thr;
        if (peak && r > 0) {
#pragma unroll
            for (int d = 0; d < 9; ++d) {
                const int ii = i + d / 3 - 1, jj = j + d % 3 - 1;
                if (d == 4 || ii < 0 || ii >= nrows || jj < 0 || jj >= nlon) continue;
                const T y = v[(int64_t)ii * nlon + jj];
                if (y > x || (y == x && d < 4)) peak = false;
            }
        }
        unsigned left = __ballot_sync(0xffffffffu, peak && r > 1);
        for (; left; left &= left - 1) {
            const int src = __ffs(left) - 1;
            const int64_t pc = __shfl_sync(0xffffffffu, p, src);
            const T xc = __shfl_sync(0xffffffffu, x, src);
            const int ic = __shfl_sync(0xffffffffu, i, src), jc = __shfl_sync(0xffffffffu, j, src);
            // windows of at most 16 columns take two rows at a time
            const int jlo = max(0, jc - r), jhi = (int)min((int64_t)nlon - 1, (int64_t)jc + r);
            const int ihi = (int)min((int64_t)nrows - 1, (int64_t)ic + r), two = r <= 7 ? 1 : 0;
            bool beaten = false;
            for (int i0 = max(0, ic - r); i0 <= ihi && !beaten; i0 += 2 << two) {
                bool b = false;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int ii = two ? i0 + 2 * u + (lane >> 4) : i0 + u;
                    if (ii > ihi) continue;
                    const T *row = v + (int64_t)ii * nlon;
                    for (int jj = jlo + (two ? lane & 15 : lane); jj <= jhi; jj += 32) {
                        const T y = row[jj];
                        b = b || y > xc || (y == xc && (int64_t)ii * nlon + jj < pc);
                    }
                }
                beaten = __any_sync(0xffffffffu, b);
            }
            if (beaten && lane == src) peak = false;
        }
        if (peak) {
            const int k = atomicAdd(count, 1);
            if (k < cap) cand[k] = p;
        }
    }
}

// Order-preserving map of a finite or infinite double onto integers; -0 and 0
// are equal.
__device__ __forceinline__ unsigned long long sort_key(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x == 0.0 ? 0.0 : x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// One CTA: bitonic sort of min(count, cap) candidates (cap a power of two <=
// kDetectCap) by (value desc, index asc), over the next power of two; the first
// max_peaks become peak records. The values are compared as integers: FP64
// comparisons at 1/64 of the rate took 1.5 us a stage (102 us for any number of
// candidates; for about 1000 of them now 39, and 16 where at most 16 peaks are
// picked instead).
template <typename T>
__global__ void __launch_bounds__(1024) k_detect_sort(const T *__restrict__ v, const int *count, const int64_t *cand,
                                                      int cap, int max_peaks, GridDev g, const GridStep *step,
                                                      DetectPeak *out)
{
    __shared__ unsigned long long sv[kDetectCap];
    __shared__ int64_t si[kDetectCap];
    const int n = min(*count, cap);
    int size = 2;
    while (size < n) size <<= 1;
    for (int t = threadIdx.x; t < size && t < cap; t += blockDim.x) {
        if (t < n) {
            si[t] = cand[t];
            sv[t] = sort_key((double)v[cand[t]]);
        } else {
            si[t] = INT64_MAX;
            sv[t] = 0ull;  // after every value's key
        }
    }
    __syncthreads();
    if (max_peaks <= 16) {
        // a few peaks are picked one by one: the sort's stages take longer
        __shared__ unsigned long long wv[32];
        __shared__ int64_t wi[32];
        __shared__ int64_t pick[16];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int r = 0; r < min(n, max_peaks); ++r) {
            unsigned long long bv = 0ull;
            int64_t bi = INT64_MAX;
            for (int t = threadIdx.x; t < n; t += blockDim.x) {
                const unsigned long long v1 = sv[t];
                const int64_t i1 = si[t];
                if (v1 > bv || (v1 == bv && i1 < bi)) {
                    bv = v1;
                    bi = i1;
                }
            }
            for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) {
                    const unsigned long long v1 = __shfl_xor_sync(0xffffffffu, bv, d);
                    const int64_t i1 = __shfl_xor_sync(0xffffffffu, bi, d);
                    if (v1 > bv || (v1 == bv && i1 < bi)) {
                        bv = v1;
                        bi = i1;
                    }
                }
                if (pass == 0) {
                    if (lane == 0) {
                        wv[warp] = bv;
                        wi[warp] = bi;
                    }
                    __syncthreads();
                    bv = wv[lane];  // every warp reduces the 32 warps' bests
                    bi = wi[lane];
                }
            }
            if (threadIdx.x == 0) pick[r] = bi;
            for (int t = threadIdx.x; t < n; t += blockDim.x)
                if (si[t] == bi) {
                    sv[t] = 0ull;  // out of the running
                    si[t] = INT64_MAX;
                }
            __syncthreads();
        }
        if (threadIdx.x < min(n, max_peaks)) si[threadIdx.x] = pick[threadIdx.x];
        __syncthreads();
        size = 0;  // sorted
    }
    for (int k = 2; k <= size && size <= cap; k <<= 1)
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            for (int w = threadIdx.x; w < size / 2; w += blockDim.x) {
                const int t = 2 * w - (w & (jj - 1)), u = t ^ jj;  // the pair of t without bit jj
                const unsigned long long vt = sv[t], vu = sv[u];
                const int64_t it = si[t], iu = si[u];
                // "a before b": larger value, or equal value and lower index
                const bool t_first = vt > vu || (vt == vu && it < iu);
                if (((t & k) == 0) != t_first) {
                    sv[t] = vu;
                    sv[u] = vt;
                    si[t] = iu;
                    si[u] = it;
                }
            }
            __syncthreads();
        }
    const GridStep st = *step;
    for (int t = threadIdx.x; t < min(n, max_peaks); t += blockDim.x) {
        const int i = g.row0 + (int)(si[t] / g.nlon), j = (int)(si[t] % g.nlon);
        double lat, lon;
        grid_node(g, st, i, j, lat, lon);
        out[t].index = si[t];
        out[t].i = i;
        out[t].j = j;
        out[t].lat_rad = lat;
        out[t].lon_rad = lon;
        out[t].value = (double)v[si[t]];
    }
}

cudaError_t launch_detect(const void *v, int prec, const GridDev &g, const GridStep *step, double thr, int r, int cap,
                          int max_peaks, int *count, int64_t *cand, DetectPeak *out, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    const int64_t G = (int64_t)g.nrows * g.nlon;
    int64_t blocks = (G + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    if (prec == DG_PREC_FP64) {
        k_detect_mark<double><<<(unsigned)blocks, 256, 0, s>>>((const double *)v, g.nrows, g.nlon, thr, r, cap, count, cand);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_detect_sort<double><<<1, 1024, 0, s>>>((const double *)v, count, cand, cap, max_peaks, g, step, out);
    } else {
        k_detect_mark<float><<<(unsigned)blocks, 256, 0, s>>>((const float *)v, g.nrows, g.nlon, thr, r, cap, count, cand);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_detect_sort<float><<<1, 1024, 0, s>>>((const float *)v, count, cand, cap, max_peaks, g, step, out);
    }
    return cudaGetLastError();
}

}  // namespace dg
