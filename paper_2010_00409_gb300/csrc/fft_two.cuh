// float32 transforms of axis lengths N = R1 R2 (both radices at most 32) with the
// radices, the tile and every shared-memory offset fixed at compile time: the
// two-pass case of fft_mixed.cuh, whose passes this file repeats in the same
// arithmetic order without the run-time index arithmetic.  At run time that arithmetic
// (divisions of the item index, strides, the dispatch over radices) was a third to a
// half of the instructions (58, 87 and 138 a value for the x, y and k-space passes of
// a 180 x 135 x 150 box against 39, 57 and 109 here), and with 24 warps an SM the
// passes were bound by instruction issue and not by memory.  Measured on that box
// (350 MB a pass), run-time passes against these: x 78 -> 59 us (5.9 TB/s), y 97 ->
// 69 us, k-space 147 -> 126 us.
//
//   cols    y or z: 16 x-columns (128 bytes a row) by R1 threads, one item of each
//           pass a thread
//   rows    x: as many rows as give 256 threads at R1 a row
//   kspace  z forward, the per-mode update, z inverse for the six components of 8
//           x-columns at one y, the spectra kept digit-reversed in shared memory
//
// Lengths: those to 1024 whose plan has two passes, of radices up to 16 where that is
// enough (two_pass_entry).  Beyond 16 points a thread takes up to 128 registers, which
// the run-time passes pay as well: 162^3 step 666 -> 530 us, 384 x 320 x 288 4.74 ->
// 3.68 ms, 480 x 400 x 360 10.2 -> 7.2 ms.  Two limits: the 16-column tile of y and z
// stops at 96 KB (900 points leave one block an SM: 228 us a pass of a 100 x 900 x 100
// box, 220 us with the run-time passes' 8 columns), the k-space tile at 226 KB (588
// points).
// float64 stays with the run-time passes: it is bound by the float64 pipe.
#pragma once

#include "fft_mixed.cuh"
#include "mode_update.cuh"

namespace psatd {

// The lengths of two radices up to 16 (index, R1, R2), for the batched advance's tiles.
#define PSATD_TWO_PAIRS(X) \
    X(0, 6, 3) X(1, 5, 4) X(2, 6, 4) X(3, 5, 5) X(4, 9, 3) X(5, 6, 5) X(6, 8, 4) X(7, 6, 6) X(8, 8, 5) \
    X(9, 9, 5) X(10, 8, 6) X(11, 10, 5) X(12, 9, 6) X(13, 10, 6) X(14, 8, 8) X(15, 9, 8) X(16, 15, 5) \
    X(17, 10, 8) X(18, 9, 9) X(19, 10, 9) X(20, 12, 8) X(21, 10, 10) X(22, 12, 9) X(23, 12, 10) X(24, 16, 8) \
    X(25, 15, 9) X(26, 12, 12) X(27, 15, 10) X(28, 16, 10) X(29, 15, 12) X(30, 16, 12) X(31, 15, 15) \
    X(32, 16, 15) X(33, 16, 16)

// The index of a plan's pair in that list, or -1.
inline int two_pair_index(const AxisPlan& pl) {
    if (pl.npass != 2) return -1;
#define PSATD_TWO_CASE(i, r1, r2) \
    if (pl.radix[0] == r1 && pl.radix[1] == r2) return i;
    PSATD_TWO_PAIRS(PSATD_TWO_CASE)
#undef PSATD_TWO_CASE
    return -1;
}
// Rows a block of 256 threads takes at once along x.
inline int two_rows_per_tile(const AxisPlan& pl) { return 256 / pl.radix[0]; }

struct TwoPassArgs {
    float2* data;
    const float2* tp;                       // position-ordered twiddles, W_N^{jk} at k R2 + j
    int axis, Nx, Ny, Nz, ncomp;
};
struct TwoPassModes {
    const float *kx, *ky, *kz;
    const ModeCoef<float>* coef;
    int mode;
    float scale;
};
struct TwoPassEntry {
    int N, R1;
    int cols_threads, cols_smem, rows_threads, rows_per_block, rows_smem;
    int kspace_threads, kspace_smem;        // 0: the six components' tile does not fit
    void (*cols[2])(TwoPassArgs);           // forward, inverse (null: tile too large, or
    void (*rows[2])(TwoPassArgs);           // a length that always takes another kernel)
    void (*kspace)(TwoPassArgs, TwoPassModes);
};
// The kernels of length N, or null.
const TwoPassEntry* two_pass_entry(int N);

#ifdef __CUDACC__
constexpr int kTwoW = 16, kTwoKW = 8;

template <int R1, int R2> struct TwoCfg {
    static constexpr int N = R1 * R2;
    static_assert(R1 >= R2, "the first radix is the larger");
    // registers a thread the register DFTs of the larger radix need
    static constexpr int regs = R1 <= 12 ? 64 : (R1 <= 16 ? 80 : (R1 <= 20 ? 96 : 128));
    static constexpr int blocks(int threads, int smem) {
        const int by_regs = 65536 / regs / threads, by_smem = 220 * 1024 / (smem + 1024);
        return by_regs < 1 || by_smem < 1 ? 1 : (by_regs < by_smem ? by_regs : by_smem);
    }
    static constexpr int cols_threads = (R1 * kTwoW + 31) / 32 * 32;
    static constexpr int cols_smem = N * kTwoW * (int)sizeof(float2);
    static constexpr bool cols = cols_smem < 96 * 1024 && N != 512;     // (512: fft_three.cu)
    static constexpr int G = 256 / R1;                                  // rows per block
    static constexpr bool rows = N != 64 && N != 128 && N != 256 && N != 512;   // (fft_fast.cu)
    static constexpr int rows_threads = (G * R1 + 31) / 32 * 32;
    static constexpr int run = R2 | 1, P = (R1 * run) | 1;              // row layout of fft_mixed.cuh
    static constexpr int rows_smem = G * P * (int)sizeof(float2);
    // k-space: 256 threads where three or more tiles share an SM, else as many as keep it busy
    static constexpr int kspace_smem = 6 * N * kTwoKW * (int)sizeof(float2);
    static constexpr bool kspace = kspace_smem <= 226 * 1024;
    static constexpr int kspace_threads = kspace_smem <= 75 * 1024 ? 256 : 512;
    // Blocks an SM: four of 256 threads (64 registers) to 120 points with radices up to
    // 12, k-space pass of 192 x 192 x 96 110 -> 102 us, 180 x 150 x 108 86 -> 82 us,
    // 180 x 180 x 120 127 -> 121 us against three; at 144 points four tiles take all of
    // the SM's shared memory from its L1 (144^3 101 -> 108 us).
    static constexpr int kspace_blocks =
        kspace_threads == 256 ? (R1 <= 12 && N <= 120 ? 4 : 3) : (R1 <= 16 ? 2 : 1);
};

// multiply v[k] by the position-ordered twiddles W_N^{jk} (conjugated for S > 0)
template <int S, int R1, int R2>
__device__ __forceinline__ void two_twiddle(float2 (&v)[R1], const float2* __restrict__ tp, int j) {
    static_for<1, R1>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const float2 w = tp[PSATD_IX(k * R2 + j, R1 * R2)];
        v[k] = S < 0 ? cmul(v[k], w) : cmulc(v[k], w);
    });
}

// CG: loads of the field go around L1 (values other SMs wrote during this launch).
template <bool CG> __device__ __forceinline__ float2 two_load(const GBuf<float2>& F, const float2* p, size_t i) {
    if constexpr (CG) return __ldcg(&F.at(p, i));
    else return F.at(p, i);
}

// One column tile: lane c of kTwoW on column base (its pointer), t = 0 .. R1 - 1.
template <int R1, int R2, int S, bool CG>
__device__ __forceinline__ void two_cols_tile(float2* base, size_t stride, int t, int c, bool col,
                                              const float2* __restrict__ tp, float2* sm, const GBuf<float2>& F) {
    constexpr int W = kTwoW;
    if (col && t < R2) {
        float2 v[R1];
        const float2* p = base + t * stride;
        static_for<0, R1>([&](auto rc) {
            v[decltype(rc)::value] = two_load<CG>(F, p, 0);
            p += R2 * stride;
        });
        reg_dft<float, S, R1>(v);
        two_twiddle<S, R1, R2>(v, tp, t);
        static_for<0, R1>([&](auto rc) { sm[(decltype(rc)::value * R2 + t) * W + c] = v[decltype(rc)::value]; });
    }
    __syncthreads();
    if (col && t < R1) {
        float2 v[R2];
        static_for<0, R2>([&](auto rc) { v[decltype(rc)::value] = sm[(t * R2 + decltype(rc)::value) * W + c]; });
        reg_dft<float, S, R2>(v);
        float2* p = base + t * stride;
        static_for<0, R2>([&](auto rc) {
            F.at(p, 0) = v[decltype(rc)::value];
            p += R1 * stride;
        });
    }
}

// nrow <= TwoCfg::G consecutive rows at base.
template <int R1, int R2, int S, bool CG>
__device__ __forceinline__ void two_rows_tile(float2* base, int nrow, const float2* __restrict__ tp, float2* sm,
                                              const GBuf<float2>& F) {
    using Cfg = TwoCfg<R1, R2>;
    constexpr int N = R1 * R2;
    const int tid = threadIdx.x;
    if (tid < nrow * R2) {
        const int w = tid / R2, j = tid - w * R2;
        const float2* p = base + w * N + j;
        float2 v[R1];
        static_for<0, R1>([&](auto rc) { v[decltype(rc)::value] = two_load<CG>(F, p, decltype(rc)::value * R2); });
        reg_dft<float, S, R1>(v);
        two_twiddle<S, R1, R2>(v, tp, j);
        float2* s = sm + w * Cfg::P + j;
        static_for<0, R1>([&](auto rc) { s[decltype(rc)::value * Cfg::run] = v[decltype(rc)::value]; });
    }
    __syncthreads();
    if (tid < nrow * R1) {
        const int w = tid / R1, u = tid - w * R1;
        const float2* s = sm + w * Cfg::P + u * Cfg::run;
        float2 v[R2];
        static_for<0, R2>([&](auto rc) { v[decltype(rc)::value] = s[decltype(rc)::value]; });
        reg_dft<float, S, R2>(v);
        float2* p = base + w * N + u;
        static_for<0, R2>([&](auto rc) { F.at(p, decltype(rc)::value * R1) = v[decltype(rc)::value]; });
    }
}

// z passes of a k-space tile (six components of kTwoKW columns, [6][position][kTwoKW] in
// sm, nw of them in the field).  The forward one ends with a barrier.
template <int R1, int R2, int TH, bool CG>
__device__ __forceinline__ void two_z_forward(const float2* base, size_t plane, size_t cstride, int nw,
                                              const float2* __restrict__ tp, float2* sm, const GBuf<float2>& F) {
    constexpr int W = kTwoKW, SLOT = R1 * R2 * W;
#pragma unroll 1
    for (int i = threadIdx.x; i < 6 * R2 * W; i += TH) {
        const int c = i % W, u = i / W, q = u / R2, j = u - q * R2;
        if (c >= nw) continue;
        const float2* p = base + q * cstride + j * plane + c;
        float2 v[R1];
        static_for<0, R1>([&](auto rc) {
            v[decltype(rc)::value] = two_load<CG>(F, p, 0);
            p += R2 * plane;
        });
        reg_dft<float, -1, R1>(v);
        two_twiddle<-1, R1, R2>(v, tp, j);
        float2* s = sm + q * SLOT + j * W + c;
        static_for<0, R1>([&](auto rc) { s[decltype(rc)::value * R2 * W] = v[decltype(rc)::value]; });
    }
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x; i < 6 * R1 * W; i += TH) {
        const int c = i % W, u = i / W;                           // u = q R1 + k1: runs of R2 positions
        if (c >= nw) continue;
        float2* s = sm + u * (R2 * W) + c;
        float2 v[R2];
        static_for<0, R2>([&](auto rc) { v[decltype(rc)::value] = s[decltype(rc)::value * W]; });
        reg_dft<float, -1, R2>(v);
        static_for<0, R2>([&](auto rc) { s[decltype(rc)::value * W] = v[decltype(rc)::value]; });
    }
    __syncthreads();
}

template <int R1, int R2, int TH>
__device__ __forceinline__ void two_z_inverse(float2* base, size_t plane, size_t cstride, int nw,
                                              const float2* __restrict__ tp, float2* sm, const GBuf<float2>& F) {
    constexpr int W = kTwoKW, SLOT = R1 * R2 * W;
#pragma unroll 1
    for (int i = threadIdx.x; i < 6 * R1 * W; i += TH) {
        const int c = i % W, u = i / W;
        if (c >= nw) continue;
        float2* s = sm + u * (R2 * W) + c;
        float2 v[R2];
        static_for<0, R2>([&](auto rc) { v[decltype(rc)::value] = s[decltype(rc)::value * W]; });
        reg_dft<float, +1, R2>(v);
        static_for<0, R2>([&](auto rc) { s[decltype(rc)::value * W] = v[decltype(rc)::value]; });
    }
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x; i < 6 * R2 * W; i += TH) {
        const int c = i % W, u = i / W, q = u / R2, j = u - q * R2;
        if (c >= nw) continue;
        const float2* s = sm + q * SLOT + j * W + c;
        float2 v[R1];
        static_for<0, R1>([&](auto rc) { v[decltype(rc)::value] = s[decltype(rc)::value * R2 * W]; });
        two_twiddle<+1, R1, R2>(v, tp, j);
        reg_dft<float, +1, R1>(v);
        float2* p = base + q * cstride + j * plane + c;
        static_for<0, R1>([&](auto rc) {
            F.at(p, 0) = v[decltype(rc)::value];
            p += R2 * plane;
        });
    }
}

template <int R1, int R2, int S>
__global__ void __launch_bounds__(TwoCfg<R1, R2>::cols_threads,
                                  TwoCfg<R1, R2>::blocks(TwoCfg<R1, R2>::cols_threads, TwoCfg<R1, R2>::cols_smem))
two_cols_kernel(const __grid_constant__ TwoPassArgs a) {
    constexpr int W = kTwoW;
    extern __shared__ __align__(16) unsigned char two_smem[];
    float2* sm = reinterpret_cast<float2*>(two_smem);             // [position][W]
    const unsigned ntile = (unsigned)(a.Nx + W - 1) / W, outer = a.axis == 1 ? a.Nz : a.Ny;
    const unsigned rest = blockIdx.x / ntile, x0 = (blockIdx.x - rest * ntile) * W;
    const unsigned comp = rest / outer, o = rest - comp * outer;
    const size_t plane = (size_t)a.Nx * a.Ny, stride = a.axis == 1 ? (size_t)a.Nx : plane;
    const unsigned c = threadIdx.x % W, t = threadIdx.x / W;
    float2* base = a.data + comp * plane * a.Nz + (a.axis == 1 ? o * plane : (size_t)o * a.Nx) + x0 + c;
    const GBuf<float2> F{a.data, (long long)a.ncomp * plane * a.Nz};
    pdl_launch_dependents();
    pdl_wait();
    two_cols_tile<R1, R2, S, false>(base, stride, (int)t, (int)c, x0 + c < (unsigned)a.Nx, a.tp, sm, F);
}

template <int R1, int R2, int S>
__global__ void __launch_bounds__(TwoCfg<R1, R2>::rows_threads,
                                  TwoCfg<R1, R2>::blocks(TwoCfg<R1, R2>::rows_threads, TwoCfg<R1, R2>::rows_smem))
two_rows_kernel(const __grid_constant__ TwoPassArgs a) {
    constexpr int N = R1 * R2, G = TwoCfg<R1, R2>::G;
    extern __shared__ __align__(16) unsigned char two_smem[];
    const long long rows = (long long)a.ncomp * a.Nz * a.Ny, row0 = (long long)blockIdx.x * G;
    const int nrow = (int)min((long long)G, rows - row0);
    pdl_launch_dependents();
    pdl_wait();
    two_rows_tile<R1, R2, S, false>(a.data + row0 * N, nrow, a.tp, reinterpret_cast<float2*>(two_smem),
                                    GBuf<float2>{a.data, rows * N});
}

template <int R1, int R2>
__global__ void __launch_bounds__(TwoCfg<R1, R2>::kspace_threads, TwoCfg<R1, R2>::kspace_blocks)
two_kspace_kernel(const __grid_constant__ TwoPassArgs a, const __grid_constant__ TwoPassModes md) {
    constexpr int W = kTwoKW, N = R1 * R2, SLOT = N * W, TH = TwoCfg<R1, R2>::kspace_threads;
    extern __shared__ __align__(16) unsigned char two_smem[];
    float2* F = reinterpret_cast<float2*>(two_smem);              // [6][position][W]
    const int Nx = a.Nx, Ny = a.Ny, tid = threadIdx.x;
    const unsigned ntile = (unsigned)(Nx + W - 1) / W;
    const int y = (int)(blockIdx.x / ntile), x0 = (int)(blockIdx.x - y * ntile) * W;
    const size_t plane = (size_t)Nx * Ny, cstride = plane * N;
    float2* base = a.data + (size_t)y * Nx + x0;
    const GBuf<float2> G{a.data, 6LL * (long long)cstride};
    const int nw = min(W, Nx - x0);
    pdl_launch_dependents();
    pdl_wait();
    two_z_forward<R1, R2, TH, false>(base, plane, cstride, nw, a.tp, F, G);

    // the update of every mode: position k1 R2 + k2 holds k_z = k1 + R1 k2
    const int Nxh = Nx / 2 + 1, Nyh = Ny / 2 + 1, ay = min(y, Ny - y);
    const float kyv = md.ky[PSATD_IX(y, Ny)];
    const bool spectral = md.mode == KS_ROTATE_SPECTRAL || md.mode == KS_ROTATE_SPECTRAL_PROJ;
#pragma unroll 1
    for (int e = tid; e < SLOT; e += TH) {
        const int c = e % W, pos = e / W, k1 = pos / R2, n = k1 + (pos - k1 * R2) * R1;
        if (c >= nw) continue;
        const int ix = x0 + c, ax = min(ix, Nx - ix), az = min(n, N - n);
        const ModeCoef<float> m =
            md.coef[PSATD_IX(((size_t)az * Nyh + ay) * Nxh + ax, (long long)(N / 2 + 1) * Nyh * Nxh)];
        const float nx = md.kx[PSATD_IX(ix, Nx)] * m.kinv, ny = kyv * m.kinv, nz = md.kz[PSATD_IX(n, N)] * m.kinv;
        float2 f[6];
        static_for<0, 6>([&](auto qc) { f[decltype(qc)::value] = F[decltype(qc)::value * SLOT + e]; });
        mode_update<float>(&f[0], &f[1], &f[2], &f[3], &f[4], &f[5], nx, ny, nz, m.C, m.S, md.mode, md.scale);
        if (spectral) {                                           // stored in natural order
            float2* p = base + n * plane + c;
            static_for<0, 6>([&](auto qc) {
                G.at(p, 0) = f[decltype(qc)::value];
                p += cstride;
            });
        } else {
            static_for<0, 6>([&](auto qc) { F[decltype(qc)::value * SLOT + e] = f[decltype(qc)::value]; });
        }
    }
    if (spectral) return;
    __syncthreads();

    two_z_inverse<R1, R2, TH>(base, plane, cstride, nw, a.tp, F, G);
}

template <int R1, int R2> TwoPassEntry two_pass_make() {
    using Cfg = TwoCfg<R1, R2>;
    TwoPassEntry e{};
    e.N = R1 * R2;
    e.R1 = R1;
    e.cols_threads = Cfg::cols_threads;
    e.cols_smem = Cfg::cols_smem;
    e.rows_threads = Cfg::rows_threads;
    e.rows_per_block = Cfg::G;
    e.rows_smem = Cfg::rows_smem;
    if constexpr (Cfg::cols) {
        e.cols[0] = two_cols_kernel<R1, R2, -1>;
        e.cols[1] = two_cols_kernel<R1, R2, +1>;
    }
    if constexpr (Cfg::rows) {
        e.rows[0] = two_rows_kernel<R1, R2, -1>;
        e.rows[1] = two_rows_kernel<R1, R2, +1>;
    }
    if constexpr (Cfg::kspace) {
        e.kspace_threads = Cfg::kspace_threads;
        e.kspace_smem = Cfg::kspace_smem;
        e.kspace = two_kspace_kernel<R1, R2>;
    }
    return e;
}
#endif

// The entries of one translation unit each (fft_two_*.cu).
const TwoPassEntry* two_pass_part0(int N);
const TwoPassEntry* two_pass_part1(int N);
const TwoPassEntry* two_pass_part2(int N);
const TwoPassEntry* two_pass_part3(int N);
const TwoPassEntry* two_pass_part4(int N);
const TwoPassEntry* two_pass_part5(int N);
const TwoPassEntry* two_pass_part6(int N);
const TwoPassEntry* two_pass_part7(int N);

}  // namespace psatd
