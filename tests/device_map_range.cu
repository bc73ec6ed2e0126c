// Lookups in delay-Doppler tables that do not hold a node's lag or bin
// (csrc/dg_map.cu): prints the error word of each case (test_gpu_map_range.py). The
// tables are as large as their shape says, so nothing is read outside of them.
#include "dg_map.cu"

#include <cstdio>
#include <cstring>
#include <vector>

using namespace dg;

template <typename T> static T *upload(const std::vector<T> &v)
{
    T *p = nullptr;
    if (cudaMalloc((void **)&p, sizeof(T) * v.size()) != cudaSuccess) std::exit(2);
    if (cudaMemcpy(p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice) != cudaSuccess) std::exit(2);
    return p;
}

int main()
{
    // receivers in one place at rest: every node has D = 0 and FDOA 0
    const int n = 64, Q = 12, NLpad = 32;
    const int64_t G = (int64_t)n * n;
    std::vector<double> xyz(3 * G, 0.0), eph(12, 0.0);
    for (int64_t p = 0; p < G; ++p) xyz[p] = 6.4e6, xyz[G + p] = 100.0 * (double)p;
    eph[0] = eph[6] = 7.0e6;
    std::vector<float> ephf(24, 0.f);
    ephf[0] = ephf[12] = 7.0e6f;
    StepDesc sd{};
    sd.n = 1000;
    MapArgs a{};
    a.sd = upload(std::vector<StepDesc>{sd});
    a.xyz = upload(xyz);
    a.eph = upload(eph);
    a.ephf = upload(ephf);
    a.fsc_hi = 0.04f;
    a.ilf_hi = 1e-6f;
    a.fs = 1e7;
    a.lambda = 0.2;
    a.G = G;
    a.nrows = a.nlon = n;
    a.S = a.ksd = a.nreg = 1;
    a.Q = Q;
    a.NLpad = NLpad;
    a.first = 1;
    a.X = upload(std::vector<float2>((size_t)Q * NLpad, make_float2(1.f, 0.f)));
    a.out = upload(std::vector<float>(G, 0.f));
    a.err = upload(std::vector<unsigned>(1, 0u));
    std::vector<float> fit(kPolyTerms * kPolyPts, 0.f);  // constant polynomials: the mean of the samples
    for (int i = 0; i < kPolyPts; ++i) fit[i] = 1.f / kPolyPts;
    a.fit = upload(fit);
    for (int poly = 0; poly < 3; ++poly)
        for (int delay : {DG_DELAY_INTEGER, DG_DELAY_LAGRANGE4}) {
            struct {
                int L0, NL;  // lag 0 at -L0 of NL
                float bin;   // and its bin coordinate
            } cases[] = {{-4, 9, 5.f}, {0, 9, 5.f}, {-8, 9, 5.f}, {1, 9, 5.f}, {-9, 9, 5.f},
                         {-4, 9, 2.01f}, {-4, 9, 8.99f}, {-4, 9, 0.4f}, {-4, 9, 10.6f}, {-300, 9, 5.f}};
            std::printf("%d %d", poly, delay);
            for (const auto &t : cases) {
                MapSnap ms{};
                ms.L0 = t.L0;
                ms.NL = t.NL;
                ms.inv_delta = 1e6f;
                ms.nu0_hi = -t.bin / ms.inv_delta;
                a.snap = upload(std::vector<MapSnap>{ms});
                a.delay = delay;
                a.poly.rows = poly == 0 ? 0 : poly == 1 ? 32 : 64;
                const size_t tiles = poly ? (size_t)(n / a.poly.rows) * (n / kPolyCols) : 1;
                a.coef = upload(std::vector<float>(tiles * kPolyStride, 0.f));
                cudaMemset(a.err, 0, sizeof(unsigned));
                if (poly && launch_map_poly(a, 0) != cudaSuccess) return 2;
                if (launch_map_lookup(a, 0) != cudaSuccess) return 2;
                unsigned e = 99;
                if (cudaMemcpy(&e, a.err, sizeof e, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
                std::printf(" %u", e);
                cudaFree((void *)a.snap);
                cudaFree(a.coef);
            }
            std::printf("\n");
        }
    return 0;
}
