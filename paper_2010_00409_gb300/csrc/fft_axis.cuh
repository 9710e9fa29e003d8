// Generic in-place FFT along one axis of a [ncomp][Nz][Ny][Nx] complex array
// (the 3D DFT of Sec. 2.1 is three of these; the kernel is exp(-ikx) forward):
// the in-place mixed-radix passes of fft_mixed.cuh over a tile of pencils.
//  - x (contiguous): W consecutive rows a block;
//  - y / z (strided): W consecutive x-columns at one (comp, z) or (comp, y), 128
//    contiguous bytes a row.
// Bound by memory traffic (one read and one write of the field): with two passes
// a block keeps its whole tile's loads in flight at once (one value per register
// of the first pass) and touches shared memory twice per value.  The staged
// radix-2/3/4/5/8 passes it replaced (three or four passes between two shared
// buffers) took 160 us along x and y of a 180 x 135 x 150 box in float32 (350 MB),
// this one 78 and 97 us, the compile-time kernels of fft_two.cuh 59 and 69 us.
#pragma once

#include "fft_mixed.cuh"

namespace psatd {

namespace {

constexpr int kThreads = 256;
// largest tile: 64 KB (three blocks an SM share its memory; their registers allow two or
// three in float32), 100 KB in float64 (two)
template <typename T> constexpr int axis_tile_cap() { return (sizeof(T) == 8 ? 100 : 64) * 1024; }

// narrow plans (radices to 16): three blocks of 256 threads per SM in float32
template <typename T, int MAXR> constexpr int axis_min_blocks() {
    return sizeof(T) == 4 ? (MAXR <= kNarrow ? 3 : 2) : (MAXR <= kNarrow ? 2 : 1);
}

template <typename T, int S, int MAXR, bool ROWS, bool PAD>
__global__ void __launch_bounds__(kThreads, axis_min_blocks<T, MAXR>())
fft_axis_kernel(cplx<T>* __restrict__ data, int axis, int Nx, int Ny, int Nz, int ncomp, int W, int logw,
                const __grid_constant__ AxisPlan pl, const cplx<T>* __restrict__ tp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* sm = reinterpret_cast<cplx<T>*>(smem_raw);
    MixTile<T> t;
    t.nq = 1;
    t.cstride = 0;
    t.slot = 0;
    t.logw = logw;
    const long long plane = (long long)Nx * Ny;
    t.buf = GBuf<cplx<T>>{data, ncomp * plane * Nz};
    if constexpr (ROWS) {
        const long long rows = (long long)ncomp * Nz * Ny, row0 = (long long)blockIdx.x * W;
        t.base = data + row0 * Nx;
        t.stride = 1;
        t.nw = (int)min((long long)W, rows - row0);
        const int n = Nx / pl.radix[0];                                 // values of a run
        t.run = PAD ? row_run_padded(pl) : row_run(Nx, pl.radix[0]);
        t.P = pl.radix[0] * t.run | 1;
        t.gap = t.run - n - (PAD ? n / pl.radix[2] : 0);
    } else {
        const unsigned ntile = (unsigned)(Nx + W - 1) >> logw, outer = axis == 1 ? Nz : Ny;
        const unsigned rest = blockIdx.x / ntile, tile = blockIdx.x - rest * ntile;
        const int comp = (int)(rest / outer), o = (int)(rest - comp * outer), x0 = (int)tile * W;
        t.base = data + comp * plane * Nz + (axis == 1 ? o * plane : (long long)o * Nx) + x0;
        t.stride = axis == 1 ? Nx : plane;
        t.nw = min(W, Nx - x0);
        t.P = t.run = t.gap = 0;
    }
    pdl_launch_dependents();
    pdl_wait();
    mix_transform<T, S, MAXR, ROWS, false, PAD>(t, sm, pl, tp);
}

}  // namespace

// Share of a float64 column pass's lanes that hold an item: W-column tiles over Nx
// columns, each pass's W N / R items in whole warps.
inline double lane_share(const AxisPlan& pl, int Nx, int W) {
    double warps = 0;
    for (int p = 0; p < pl.npass; ++p) {
        const int items = W * (pl.N / pl.radix[p]);
        warps += (double)((items + 31) / 32 * 32) / items;
    }
    return (double)Nx / ((Nx + W - 1) / W * W) * pl.npass / warps;
}

// Lanes a float64 row pass of W rows spends per value's item, each pass in whole warps;
// with two passes or fewer half of it counted in rounds of all 256 threads (an uneven
// last round leaves warps idle; three short passes with two blocks an SM hide that).
inline double row_cost(const AxisPlan& pl, int W) {
    double c = 0;
    for (int p = 0; p < pl.npass; ++p) {
        const int items = W * (pl.N / pl.radix[p]);
        const double warps = (items + 31) / 32 * 32, rounds = items > 256 ? (items + 255) / 256 * 256 : warps;
        c += (pl.npass > 2 ? warps : 0.5 * (warps + rounds)) / items;
    }
    return c;
}

// Tile of the transform along an axis: W pencils (a power of two of x-columns, 128
// contiguous bytes a row, along y and z; rows giving about 256 first-pass items
// along x), scaled by 2^shift, halved until the tile fits `cap` bytes.
template <typename T>
void mix_tile_shape(int axis, const AxisPlan& pl, int Nx, int shift, size_t cap, int* W, size_t* bytes) {
    const int es = (int)sizeof(cplx<T>), N = pl.N;
    const int row = sizeof(T) == 4 && row_padded(pl) ? pl.radix[0] * row_run_padded(pl) | 1 : row_stride(N, pl.radix[0]);
    const size_t per = (size_t)(axis == 0 ? row : N) * es;
    int w;
    if (axis == 0) {
        w = max(1, min(128, 256 * pl.radix[0] / N));
        // float64 is bound by its pipe, where idle lanes cost as much as busy ones: 1000
        // points (10 x 10 x 10) in two rows give 200 items a pass.  1000 x 64 x 64 step
        // 7.61 -> 7.32 ms, 480 x 64 x 64 3.78 -> 3.64 ms, 60 x 20 x 60 -10 %.
        if (sizeof(T) == 8) {
            int best = w;
            for (int v = max(1, w / 2); v <= 4 * w && v * per <= cap; ++v)
                if (row_cost(pl, v) < 0.97 * row_cost(pl, best)) best = v;
            w = best;
        }
    } else {
        w = 1;
        while (w < Nx && w < 128 / es) w *= 2;
        // float64 is bound by its pipe, where an idle lane costs as much as a busy one:
        // up to 32 columns where that fills the warps better (N = 20 in one pass of
        // radix 20 leaves 24 of 32 lanes idle at eight columns).  y passes of
        // 1000 x 20 x 90 1128 -> 300 us, 75 x 75 x 96 238 -> 197 us, 75 x 160 x 72 297 -> 279 us.
        // A gain under 5 % isn't worth the wider tile's fewer blocks.
        if (sizeof(T) == 8) {
            int best = w;
            for (int v = 2 * w; v <= 32 && v / 2 < Nx && v * per <= cap; v *= 2)
                if (lane_share(pl, Nx, v) > 1.05 * lane_share(pl, Nx, best)) best = v;
            w = best;
        }
    }
    if (shift > 0) w = min(axis == 0 ? 256 : 32, w << shift);
    if (shift < 0) w = max(1, w >> -shift);
    while (w > 1 && w * per > cap) w /= 2;
    *W = w;
    *bytes = w * per;
}

template <typename T>
cudaError_t launch_fft_axis(cplx<T>* data, int ncomp, const GridGeom& g, const Tables<T>& tb,
                            int axis, int dir, cudaStream_t s, long long* nlaunch) {
    const AxisPlan& pl = tb.plan[axis];
    if (pl.N <= 1) return cudaSuccess;
    int W, maxr = 0, logw = 0;
    size_t smem;
    mix_tile_shape<T>(axis, pl, g.Nx, tb.tile_shift, axis == 0 ? axis_tile_cap<T>() : 64 * 1024, &W, &smem);
    while ((1 << logw) < W) ++logw;
    for (int p = 0; p < pl.npass; ++p) maxr = max(maxr, pl.radix[p]);
    const long long nblocks = axis == 0 ? ((long long)ncomp * g.Nz * g.Ny + W - 1) / W
                                        : (long long)ncomp * (axis == 1 ? g.Nz : g.Ny) * ((g.Nx + W - 1) / W);
    if (nblocks > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
    // threads: the items of the pass with the smallest radix, at most 256
    int minr = maxr;
    for (int p = 0; p < pl.npass; ++p) minr = min(minr, pl.radix[p]);
    const long long items = (long long)W * (pl.N / minr);
    const int threads = (int)(items >= kThreads ? kThreads : (items + 31) / 32 * 32);
    auto launch = [&](auto sc, auto mc, auto rc, auto pc) {
        auto k = fft_axis_kernel<T, decltype(sc)::value, decltype(mc)::value, decltype(rc)::value, decltype(pc)::value>;
        const cudaError_t e = allow_smem<axis_tile_cap<T>()>(k);
        if (e != cudaSuccess) return e;
        if (nlaunch) ++*nlaunch;
        return launch_pdl(k, dim3((unsigned)nblocks), dim3(threads), smem, s, data, axis, g.Nx, g.Ny, g.Nz, ncomp, W,
                          logw, pl, tb.twp[axis]);
    };
    auto by_rows = [&](auto sc, auto mc) {
        if (axis != 0) return launch(sc, mc, std::false_type{}, std::false_type{});
        if constexpr (sizeof(T) == 8)                             // (wide float64 plans exist along z alone)
            return launch(sc, std::integral_constant<int, kNarrow>{}, std::true_type{}, std::false_type{});
        else
            return row_padded(pl) ? launch(sc, std::integral_constant<int, kNarrow>{}, std::true_type{}, std::true_type{})
                                  : launch(sc, mc, std::true_type{}, std::false_type{});
    };
    auto by_radix = [&](auto sc) {
        return maxr <= kNarrow ? by_rows(sc, std::integral_constant<int, kNarrow>{})
                               : by_rows(sc, std::integral_constant<int, kWide>{});
    };
    return dir < 0 ? by_radix(std::integral_constant<int, -1>{}) : by_radix(std::integral_constant<int, 1>{});
}

}  // namespace psatd
