// Fused k-space pass (generic sizes): forward FFT along z, the per-mode PSATD
// update of Eq. 3-4 (Sec. 2.1), and the inverse FFT along z, for all six
// components of a tile of W x-columns at one y.  The x and y transforms of the
// step have already been applied, so after the forward z transform the tile
// holds Fourier amplitudes E^(k), B^(k) of the modes (kx[x0..x0+W), ky[y], kz[*]).
//
// Update per mode, with C' = cos(c|k|dt)/Ntot, S' = sin(c|k|dt)/Ntot (the 1/Ntot
// of the inverse DFT folded in) and n = k/|k| (0 at k = 0):
//   E <- C' (E - n (n.E)) + i S' n x B
//   B <- C' B - i S' n x E                (both right-hand sides from step n)
// The z transforms are the in-place mixed-radix passes of fft_mixed.cuh on all six
// components at once: the first pass loads the tile, the update runs on the
// digit-reversed spectra in place, the passes run backwards for the inverse and
// the last one stores to the field, so the tile is the block's only buffer.  The
// staged small-radix passes it replaced, one component at a time with a partner
// buffer, took 581 us on a 180 x 135 x 150 box in float32, this one 147 us (126 us
// with the compile-time kernels of fft_two.cuh).
// KS_PROJECT instead removes the longitudinal part of E and B and scales by
// 1/Ntot (the one-time projection after initialisation).
#include "fft_mixed.cuh"
#include "mode_update.cuh"

namespace psatd {

namespace {

constexpr int kThreads = 256;
constexpr int kTileMax = 227 * 1024;

template <typename T, int MAXR>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? (MAXR <= kNarrow ? 3 : 2) : 1)
kspace_z_kernel(cplx<T>* __restrict__ data, int Nx, int Ny, int Nz, int W, int logw,
                const __grid_constant__ AxisPlan pl, const cplx<T>* __restrict__ tp, const T* __restrict__ kx,
                const T* __restrict__ ky, const T* __restrict__ kz, const ModeCoef<T>* __restrict__ coef, int mode,
                T scale) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* F = reinterpret_cast<cplx<T>*>(smem_raw);        // [6][Nz][W], digit-reversed kz
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int ntile = (Nx + W - 1) >> logw;
    const int y = blockIdx.x / ntile, tile = blockIdx.x - y * ntile, x0 = tile * W;
    const long long plane = (long long)Nx * Ny, cstride = plane * Nz;
    const int ct = Nz << logw;                                // one component's slot
    MixTile<T> t;
    t.base = data + (long long)y * Nx + x0;
    t.buf = GBuf<cplx<T>>{data, 6LL * cstride};
    t.cstride = cstride;
    t.stride = plane;
    t.logw = logw;
    t.nw = min(W, Nx - x0);
    t.nq = 6;
    t.slot = ct;
    t.P = t.run = t.gap = 0;
    pdl_launch_dependents();
    pdl_wait();
    mix_forward<T, MAXR, false>(t, F, pl, tp);

    const int Nxh = Nx / 2 + 1, Nyh = Ny / 2 + 1;
    const int ay = min(y, Ny - y);
    const T kyv = ky[PSATD_IX(y, Ny)];
    const bool spectral = mode == KS_ROTATE_SPECTRAL || mode == KS_ROTATE_SPECTRAL_PROJ;
    for (int e = tid; e < ct; e += nthr) {
        const int c = e & (W - 1), n = mix_frequency(pl, e >> logw);
        if (c >= t.nw) continue;
        const int ix = x0 + c;
        const int ax = min(ix, Nx - ix), az = min(n, Nz - n);
        const ModeCoef<T> m = coef[PSATD_IX(((size_t)az * Nyh + ay) * Nxh + ax, (long long)(Nz / 2 + 1) * Nyh * Nxh)];
        const T nxv = kx[PSATD_IX(ix, Nx)] * m.kinv, nyv = kyv * m.kinv, nzv = kz[PSATD_IX(n, Nz)] * m.kinv;
        cplx<T> f[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) f[q] = F[q * ct + e];
        mode_update<T>(&f[0], &f[1], &f[2], &f[3], &f[4], &f[5], nxv, nyv, nzv, m.C, m.S, mode, scale);
        if (spectral) {                                       // stored in natural order
            cplx<T>* p = t.base + n * plane + c;
#pragma unroll
            for (int q = 0; q < 6; ++q) t.buf.at(p, q * cstride) = f[q];
        } else {
#pragma unroll
            for (int q = 0; q < 6; ++q) F[q * ct + e] = f[q];
        }
    }
    if (spectral) return;
    __syncthreads();
    mix_inverse<T, MAXR>(t, F, pl, tp);
}

// The per-mode update alone, on a spectrum already transformed along all three
// axes (the z transforms run as separate launches for axis lengths without a
// fused kernel): one thread per mode, x fastest, all six components.
template <typename T>
__global__ void __launch_bounds__(kThreads)
modes_kernel(cplx<T>* __restrict__ data, int Nx, int Ny, int Nz, const T* __restrict__ kx,
             const T* __restrict__ ky, const T* __restrict__ kz, const ModeCoef<T>* __restrict__ coef, int mode,
             T scale) {
    const size_t n = (size_t)Nx * Ny * Nz;
    const int Nxh = Nx / 2 + 1, Nyh = Ny / 2 + 1;
    pdl_launch_dependents();
    pdl_wait();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const int ix = (int)(e % Nx);
        const size_t r = e / Nx;
        const int iy = (int)(r % Ny), iz = (int)(r / Ny);
        const int ax = min(ix, Nx - ix), ay = min(iy, Ny - iy), az = min(iz, Nz - iz);
        const ModeCoef<T> m = coef[PSATD_IX(((size_t)az * Nyh + ay) * Nxh + ax, (long long)(Nz / 2 + 1) * Nyh * Nxh)];
        const GBuf<cplx<T>> G{data, 6LL * (long long)n};
        mode_update<T>(&G[e], &G[n + e], &G[2 * n + e], &G[3 * n + e], &G[4 * n + e], &G[5 * n + e],
                       kx[PSATD_IX(ix, Nx)] * m.kinv, ky[PSATD_IX(iy, Ny)] * m.kinv, kz[PSATD_IX(iz, Nz)] * m.kinv,
                       m.C, m.S, mode, scale);
    }
}

}  // namespace

template <typename T>
cudaError_t launch_modes(cplx<T>* data, const GridGeom& g, const Tables<T>& tb, int mode, double scale,
                         cudaStream_t s) {
    const size_t n = (size_t)g.Nx * g.Ny * g.Nz;
    long long blocks = (long long)((n + kThreads - 1) / kThreads);
    if (blocks > 152LL * 32) blocks = 152LL * 32;
    return launch_pdl(modes_kernel<T>, dim3((unsigned)blocks), dim3(kThreads), 0, s, data, g.Nx, g.Ny, g.Nz, tb.k[0],
                      tb.k[1], tb.k[2], tb.coef, mode, (T)scale);
}

template cudaError_t launch_modes<float>(cplx<float>*, const GridGeom&, const Tables<float>&, int, double, cudaStream_t);
template cudaError_t launch_modes<double>(cplx<double>*, const GridGeom&, const Tables<double>&, int, double, cudaStream_t);

template <typename T>
cudaError_t launch_kspace_z(cplx<T>* data, const GridGeom& g, const Tables<T>& tb, int mode,
                            double scale, cudaStream_t s, long long* nlaunch) {
    const int es = (int)sizeof(cplx<T>);
    const AxisPlan& pl = tb.plan[2];
    // 64 contiguous bytes a row of the tile; the six components' tile capped at 112 KB
    // in float32 (two blocks per SM; three from 192 points down), 100 KB in float64 (two)
    auto bytes = [&](int w) { return (size_t)6 * g.Nz * w * es; };
    int W = 1;
    while (W < g.Nx && W < 64 / es) W *= 2;
    if (tb.tile_shift > 0) W <<= tb.tile_shift;
    if (tb.tile_shift < 0) W = max(1, W >> -tb.tile_shift);
    while (W > 1 && bytes(W) > (es == 8 ? 112 : 100) * 1024) W /= 2;
    const size_t smem = bytes(W);
    if (smem > kTileMax) return cudaErrorInvalidValue;
    int logw = 0, maxr = 0;
    while ((1 << logw) < W) ++logw;
    for (int p = 0; p < pl.npass; ++p) maxr = max(maxr, pl.radix[p]);
    const long long nblocks = (long long)g.Ny * ((g.Nx + W - 1) / W);
    const long long items = (long long)W * g.Nz;               // the update's
    const int threads = (int)(items >= kThreads ? kThreads : (items + 31) / 32 * 32);
    auto launch = [&](auto mc) {
        auto k = kspace_z_kernel<T, decltype(mc)::value>;
        const cudaError_t e = allow_smem<kTileMax>(k);
        if (e != cudaSuccess) return e;
        if (nlaunch) ++*nlaunch;
        return launch_pdl(k, dim3((unsigned)nblocks), dim3(threads), smem, s, data, g.Nx, g.Ny, g.Nz, W, logw, pl,
                          tb.twp[2], tb.k[0], tb.k[1], tb.k[2], tb.coef, mode, (T)scale);
    };
    return maxr <= kNarrow ? launch(std::integral_constant<int, kNarrow>{})
                           : launch(std::integral_constant<int, kWide>{});
}

template cudaError_t launch_kspace_z<float>(cplx<float>*, const GridGeom&, const Tables<float>&, int, double, cudaStream_t, long long*);
template cudaError_t launch_kspace_z<double>(cplx<double>*, const GridGeom&, const Tables<double>&, int, double, cudaStream_t, long long*);

}  // namespace psatd
