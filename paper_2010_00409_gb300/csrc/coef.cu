// The per-mode coefficient table of Eq. 3-4 (Sec. 2.1), one entry (C'/Ntot,
// S'/Ntot, 1/|k|) per octant mode (|m_z|, |m_y|, |m_x|), built on the device in
// float64 and rounded once.
//
// A step size or a one-shot time that the context has not seen needs a new
// table: 151 k entries at 96 x 108 x 108, 2.1 M at 256^3.  Each is a square
// root, a division and one sincos in float64, so the launch is bound by the
// float64 pipe (1/64 of the float32 rate); one thread per entry with x fastest
// gives 16- or 32-byte stores to consecutive addresses.  It replaced a host loop
// and an upload (about 28 ns an entry, measured as 17.2 ms for four one-shots
// of new times at 96 x 108 x 108, against 1.47 ms with this kernel).
#include "common.cuh"

namespace psatd {

namespace {

constexpr int kThreads = 256;

struct CoefGeom {
    int N[3];
    double d[3];
    double c, dt;
    int projection, slot_order;
};

template <typename T>
__global__ void __launch_bounds__(kThreads)
coef_kernel(CoefGeom g, const int* __restrict__ slot_mode, ModeCoef<T>* __restrict__ tab) {
    const int hx = g.N[0] / 2 + 1, hy = g.N[1] / 2 + 1, hz = g.N[2] / 2 + 1;
    const long long n = (long long)hx * hy * hz;
    const double ntot = (double)g.N[0] * g.N[1] * g.N[2];
    constexpr double two_pi = 6.28318530717958647692;
    for (long long e = blockIdx.x * (long long)kThreads + threadIdx.x; e < n; e += (long long)gridDim.x * kThreads) {
        const int ax = (int)(e % hx);
        const long long r = e / hx;
        const int ay = (int)(r % hy), az = (int)(r / hy);
        // slot order: column p < Nx/2 holds the x mode of half-spectrum slot p,
        // column Nx/2 the x Nyquist mode
        const int mx = (g.slot_order && ax < g.N[0] / 2) ? slot_mode[PSATD_IX(ax, g.N[0] / 2)] : ax;
        const double kx = two_pi * mx / (g.N[0] * g.d[0]);
        const double ky = two_pi * ay / (g.N[1] * g.d[1]);
        const double kz = two_pi * az / (g.N[2] * g.d[2]);
        const double km = sqrt(kx * kx + ky * ky + kz * kz);
        double sn = 0.0, cs = 1.0;
        if (!g.projection) sincos(g.c * km * g.dt, &sn, &cs);
        ModeCoef<T> m;
        m.C = (T)(cs / ntot);
        m.S = (T)(sn / ntot);
        m.kinv = (T)(km > 0.0 ? 1.0 / km : 0.0);
        m.pad = (T)0;
        tab[PSATD_IX(e, n)] = m;
    }
}

}  // namespace

template <typename T>
cudaError_t launch_coef(ModeCoef<T>* tab, const GridGeom& g, double dt, bool projection, const int* slot_mode,
                        cudaStream_t s) {
    CoefGeom cg{{g.Nx, g.Ny, g.Nz}, {g.dx, g.dy, g.dz}, g.c, dt, projection ? 1 : 0, slot_mode ? 1 : 0};
    const long long n = (long long)(g.Nx / 2 + 1) * (g.Ny / 2 + 1) * (g.Nz / 2 + 1);
    long long blocks = (n + kThreads - 1) / kThreads;
    if (blocks > (1LL << 20)) blocks = 1LL << 20;
    coef_kernel<T><<<(unsigned)blocks, kThreads, 0, s>>>(cg, slot_mode, tab);
    return cudaGetLastError();
}

template cudaError_t launch_coef<float>(ModeCoef<float>*, const GridGeom&, double, bool, const int*, cudaStream_t);
template cudaError_t launch_coef<double>(ModeCoef<double>*, const GridGeom&, double, bool, const int*, cudaStream_t);

}  // namespace psatd
