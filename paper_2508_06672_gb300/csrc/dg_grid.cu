// dg_grid.cu -- candidate grid to ECEF (Algorithm 1, first step; Sec. III)
// and the per-snapshot geometry table used for inspection (Eq. 3-10).
#include "dg_internal.cuh"

namespace dg {

// Geodetic (lat, lon, h = 0) on WGS-84 to ECEF: N = a / sqrt(1 - e2 sin^2 lat),
// x = N cos lat cos lon, y = N cos lat sin lon, z = N (1 - e2) sin lat. Output
// SoA [3][G]. A CTA takes tiles of 16 rows x 64 columns: the row's and the
// column's sines are evaluated once per tile (80 FP64 sin/cos pairs for 1024
// nodes; one per node is bound by the FP64 units, 1/64 of the FP32 rate: 15 us
// for a 41 x 41 grid on 7 SMs), and a node is two products. Every value is the
// same expression of the node's own row and column. grids (device,
// optional): grid blockIdx.y of an array, all of one size, in place of g.
// step_out (optional): the grid's angular steps, for kernels that place nodes.
constexpr int kEcefRows = 16, kEcefCols = 64;

__global__ void __launch_bounds__(256) k_grid_ecef(GridDev g, double *__restrict__ xyz, const ArgmaxResult *centre,
                                                   const GridDev *__restrict__ grids, GridStep *step_out)
{
    __shared__ double s_ncl[kEcefRows], s_z[kEcefRows], s_so[kEcefCols], s_co[kEcefCols];
    if (grids) g = grids[blockIdx.y];
    if (centre) centre_on(g, centre);
    const int64_t G = (int64_t)g.nrows * g.nlon;
    xyz += 3 * G * blockIdx.y;
    const GridStep st = grid_step(g);
    if (step_out && blockIdx.x == 0 && threadIdx.x == 0) step_out[blockIdx.y] = st;
    const double e2 = kF * (2.0 - kF);
    const int tj = (g.nlon + kEcefCols - 1) / kEcefCols, ti = (g.nrows + kEcefRows - 1) / kEcefRows;
    const int t = threadIdx.x;
    for (int64_t tile = blockIdx.x; tile < (int64_t)ti * tj; tile += gridDim.x) {
        const int r0 = (int)(tile / tj) * kEcefRows, c0 = (int)(tile % tj) * kEcefCols;
        __syncthreads();
        if (t < kEcefRows || (t >= 32 && t < 32 + kEcefCols)) {  // rows in the first warp, columns in the next two
            double lat, lon;
            grid_node(g, st, g.row0 + r0 + (t < 32 ? t : 0), c0 + (t < 32 ? 0 : t - 32), lat, lon);
            double sn, cs;
            sincos(t < 32 ? lat : lon, &sn, &cs);
            if (t < 32) {
                const double n = __ddiv_rn(kA, __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(__dmul_rn(e2, sn), sn))));
                s_ncl[t] = __dmul_rn(n, cs);
                s_z[t] = __dmul_rn(__dmul_rn(n, 1.0 - e2), sn);
            } else {
                s_so[t - 32] = sn;
                s_co[t - 32] = cs;
            }
        }
        __syncthreads();
        for (int i = t; i < kEcefRows * kEcefCols; i += 256) {
            const int r = i / kEcefCols, c = i % kEcefCols;
            if (r0 + r < g.nrows && c0 + c < g.nlon) {
                const int64_t p = (int64_t)(r0 + r) * g.nlon + c0 + c;
                xyz[p] = __dmul_rn(s_ncl[r], s_co[c]);
                xyz[G + p] = __dmul_rn(s_ncl[r], s_so[c]);
                xyz[2 * G + p] = s_z[r];
            }
        }
    }
}

cudaError_t launch_grid_ecef(const GridDev &g, double *xyz, cudaStream_t s, const ArgmaxResult *centre,
                             const GridDev *grids, int ngrids, GridStep *step_out)
{
    int64_t blocks = (int64_t)((g.nrows + kEcefRows - 1) / kEcefRows) * ((g.nlon + kEcefCols - 1) / kEcefCols);
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_grid_ecef<<<dim3((unsigned)blocks, (unsigned)ngrids), 256, 0, s>>>(g, xyz, centre, grids, step_out);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_step_geometry(int64_t G, const double *__restrict__ xyz,
                                                       const double *__restrict__ eph_k, double fs,
                                                       double lambda, int delay_mode, int *lag,
                                                       double *Dout, double *nuout)
{
    double e[12];
#pragma unroll
    for (int t = 0; t < 12; ++t) e[t] = __ldg(eph_k + t);
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < G;
         p += (int64_t)gridDim.x * blockDim.x) {
        double D, nu;
        geometry(xyz[p], xyz[G + p], xyz[2 * G + p], e, fs, lambda, D, nu);
        if (lag) lag[p] = lag_of(D, delay_mode);
        if (Dout) Dout[p] = D;
        if (nuout) nuout[p] = nu;
    }
}

cudaError_t launch_step_geometry(const GridDev &g, const double *xyz, const double *eph_k,
                                 double fs, double lambda, int delay_mode, int *lag, double *D,
                                 double *nu, cudaStream_t s)
{
    const int64_t G = (int64_t)g.nrows * g.nlon;
    int64_t blocks = (G + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_step_geometry<<<(unsigned)blocks, 256, 0, s>>>(G, xyz, eph_k, fs, lambda, delay_mode, lag, D, nu);
    return cudaGetLastError();
}

}  // namespace dg
