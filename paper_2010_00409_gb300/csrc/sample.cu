// Focal-plane sampling (Sec. 2.3, Eq. 13-16).
//
// The field at a physical point R = (x_p, y, z) is u~(T(R)) * I_S(t)(R), with T
// of Eq. 13 and u~ the exact trigonometric interpolant of the periodic grid
// field: u~(r) = (1/N) sum_m F(m) exp(i k_m . (r - r_min)).  Substituting the
// forward DFT gives the separable form
//     u~(r) = sum_{i,j,l} w_x(x - x_i) w_y(y - y_j) w_z(z - z_l) f_{l j i},
//     w_N(s) = (1/N) sum_m exp(i 2 pi m s / (N d)),  m = -floor(N/2) .. ceil(N/2)-1,
// and the geometric sum closes to
//     w_N(s) = exp(i (m_lo + (N-1)/2) phi) sin(N phi / 2) / (N sin(phi / 2)),
//     phi = 2 pi s / (N d)   (w = 1 at phi = 0; w is N d-periodic in s).
// The three contractions (x, then y, then z) run in float64 for float64
// storage and in double-float arithmetic (ff.cuh: float32 pairs, ~48 bits) for
// float32 storage, whose inputs are float32: the same sums (to about 1e-14 of the sum
// of the magnitudes over 2048 points, less over fewer) without
// float64 instructions, which GB300 issues at 1/64 of the float32 rate.  The
// weights and the partial sums g, h then live in the scratch buffers as float4
// {re.h, re.l, im.h, im.l} (the size of a double2).
#include <type_traits>

#include "common.cuh"
#include "ff.cuh"

namespace psatd {

namespace {

// The angles are kept in units of pi and reduced before the sine and cosine: one
// sincospi (no large-argument reduction) instead of a sine and a cosine of up to
// N pi radians.
__device__ __forceinline__ double2 dirichlet_weight(double s, int N, double d) {
    double u = s / (N * d);
    u -= floor(u + 0.5);                       // u in [-1/2, 1/2)
    if (u == 0.0) return make_double2(1.0, 0.0);
    const double m_c = (double)(-(N / 2)) + 0.5 * (N - 1);
    const double ratio = sinpi(N * u) / (N * sinpi(u));
    double sn, cs;
    sincospi(2.0 * m_c * u, &sn, &cs);
    return make_double2(ratio * cs, ratio * sn);
}

__device__ __forceinline__ double cut_out_indicator(double x, double y, double z, double t,
                                                    const ShellGeom& sh, double c) {
    // Eq. 15-16; the third case reads "R > r(t)" (the printed "R > l(t)" would
    // remove the focus itself, since l(t) <= 0 there).
    const double R = sqrt(x * x + y * y + z * z);
    const double Rmin = sh.R0 - 0.5 * sh.L, Rmax = sh.R0 + 0.5 * sh.L;
    const double l = -Rmax + c * t, r = -Rmin + c * t;
    bool zero = false;
    if (r < 0) zero = zero || (R >= -l) || (R < -r) || (x > 0);
    if (l <= 0 && r >= 0) {
        zero = zero || ((x < 0) && (R > sh.L));
        zero = zero || ((x >= 0) && (R > r));
    }
    if (l > 0) zero = zero || (R <= l) || (R > r) || (x < 0);
    return zero ? 0.0 : 1.0;
}

// The same with the radius in float32 where that decides: a point further than
// 1e-5 of the sum of the lengths involved from every radius the cases compare with
// takes the float32 comparisons, any other the float64 ones, so
// the decision is always the float64 one.  Four float64 evaluations a thread held
// the z contraction's last warps for about 6 us.
__device__ __forceinline__ float cut_out_f(double x, double y0, double y1, int n, int N, double z0, double z1, int m,
                                           int M, double t, const ShellGeom& sh, double c) {
    const float xf = (float)x, ct = (float)(c * t), R0 = (float)sh.R0, L = (float)sh.L;
    const float yf = (float)y0 + ((float)y1 - (float)y0) * ((float)n / (float)N);
    const float zf = (float)z0 + ((float)z1 - (float)z0) * ((float)m / (float)M);
    const float R = sqrtf(xf * xf + yf * yf + zf * zf);
    const float l = ct - (R0 + 0.5f * L), r = ct - (R0 - 0.5f * L);
    const float size = fabsf(xf) + fabsf((float)y0) + fabsf((float)y1) + fabsf((float)z0) + fabsf((float)z1) +
                       fabsf(ct) + fabsf(R0) + fabsf(L);
    const float tol = 1e-5f * size;
    const bool clear = size > 1e-12f && size < 1e15f && fabsf(l) > tol && fabsf(r) > tol &&
                       fabsf(R - fabsf(l)) > tol && fabsf(R - fabsf(r)) > tol && fabsf(R - L) > tol;
    if (!clear) {                                             // (also NaN, and squares that leave float32's range)
        const double y = y0 + (y1 - y0) * n / N, z = z0 + (z1 - z0) * m / M;
        return (float)cut_out_indicator(x, y, z, t, sh, c);
    }
    bool zero = false;
    if (r < 0.f) zero = R >= -l || R < -r || x > 0.0;
    else if (l <= 0.f) zero = x < 0.0 ? R > L : R > r;
    else zero = R <= l || R > r || x < 0.0;
    return zero ? 0.f : 1.f;
}

// a weight in float64 (double2) or double-float (float4) form
template <bool FFW>
__device__ __forceinline__ void put_w(double2* w, int i, int n, double2 v) {
    if constexpr (FFW) reinterpret_cast<float4*>(w)[PSATD_IX(i, n)] = cff_from(v.x, v.y);
    else w[PSATD_IX(i, n)] = v;
}

// Weight tid of the concatenated x, y and z weights, stored once the previous
// kernel of the stream is done with the buffers (the weights themselves depend on
// no memory, so they are computed while it finishes).  Every thread waits.
template <bool FFW>
__device__ __forceinline__ void store_weight(int tid, int nwx, int nwy, int nwz, double2 w, double2* wx, double2* wy,
                                             double2* wz) {
    pdl_launch_dependents();
    pdl_wait();
    if (tid < nwx) put_w<FFW>(wx, tid, nwx, w);
    else if (tid < nwx + nwy) put_w<FFW>(wy, tid - nwx, nwy, w);
    else if (tid < nwx + nwy + nwz) put_w<FFW>(wz, tid - nwx - nwy, nwz, w);
}

// 64 threads a block: 16.5 k weights of one sincospi each are bound by the
// float64 pipe, and blocks of 256 would leave half of the SMs' pipes idle
constexpr int kWThreads = 64;

template <bool FFW>
__global__ void weights_kernel(GridGeom g, double x_phys, int ny, int nz, double y0, double y1,
                               double z0, double z1, double2* wx, double2* wy, double2* wz) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nwx = g.Nx, nwy = ny * g.Ny, nwz = nz * g.Nz;
    double2 w = make_double2(0.0, 0.0);
    if (tid < nwx) {
        const double D = g.Nx * g.dx;
        double q = (x_phys - g.x_min) / D;
        const double xt = g.x_min + D * (q - floor(q));              // Eq. 13
        w = dirichlet_weight(xt - (g.x_min + tid * g.dx), g.Nx, g.dx);
    } else if (tid < nwx + nwy) {
        const int e = tid - nwx, p = e / g.Ny, j = e - p * g.Ny;
        const double y = y0 + (y1 - y0) * p / ny;
        w = dirichlet_weight(y - (g.y_min + j * g.dy), g.Ny, g.dy);
    } else if (tid < nwx + nwy + nwz) {
        const int e = tid - nwx - nwy, q = e / g.Nz, l = e - q * g.Nz;
        const double z = z0 + (z1 - z0) * q / nz;
        w = dirichlet_weight(z - (g.z_min + l * g.dz), g.Nz, g.dz);
    }
    store_weight<FFW>(tid, nwx, nwy, nwz, w, wx, wy, wz);
}

// Weights that evaluate the interpolant straight from a spectrum that already
// carries the 1/N of the inverse DFT (as the k-space pass leaves it):
// u~(r) = sum_m G(m) prod_a exp(i k_{a,m} (r_a - r_min,a)),  G = F / N.
__device__ __forceinline__ double2 mode_phase(int i, int N, double d, double s) {
    const int m = i <= (N - 1) / 2 ? i : i - N;
    double sn, cs;
    sincospi(2.0 * (double)m * (s / (N * d)), &sn, &cs);
    return make_double2(cs, sn);
}

template <bool FFW>
__global__ void spectral_weights_kernel(GridGeom g, double x_phys, int ny, int nz, double y0, double y1,
                                        double z0, double z1, double2* wx, double2* wy, double2* wz) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nwx = g.Nx, nwy = ny * g.Ny, nwz = nz * g.Nz;
    double2 w = make_double2(0.0, 0.0);
    if (tid < nwx) {
        const double D = g.Nx * g.dx;
        double q = (x_phys - g.x_min) / D;
        const double xt = g.x_min + D * (q - floor(q));              // Eq. 13
        w = mode_phase(tid, g.Nx, g.dx, xt - g.x_min);
    } else if (tid < nwx + nwy) {
        const int e = tid - nwx, p = e / g.Ny, j = e - p * g.Ny;
        w = mode_phase(j, g.Ny, g.dy, y0 + (y1 - y0) * p / ny - g.y_min);
    } else if (tid < nwx + nwy + nwz) {
        const int e = tid - nwx - nwy, q = e / g.Nz, l = e - q * g.Nz;
        w = mode_phase(l, g.Nz, g.dz, z0 + (z1 - z0) * q / nz - g.z_min);
    }
    store_weight<FFW>(tid, nwx, nwy, nwz, w, wx, wy, wz);
}

struct CompList { int c[6]; };

// g[a][l][j] = sum_i wx[i] f[c_a][l][j][i]; one warp per (a, l, j) row.
template <typename T>
__global__ void contract_x_kernel(const cplx<T>* __restrict__ f, GridGeom g, CompList cl, int ncomp,
                                  const double2* __restrict__ wx, double2* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long rows = (long long)ncomp * g.Nz * g.Ny;
    if (warp >= rows) return;
    const int a = (int)(warp / ((long long)g.Nz * g.Ny));
    const long long rl = warp - (long long)a * g.Nz * g.Ny;
    const cplx<T>* row = f + (size_t)cl.c[a] * g.Nx * g.Ny * g.Nz + (size_t)rl * g.Nx;
    const GBuf<const cplx<T>> F{f, 6LL * g.Nx * g.Ny * g.Nz};
    double re = 0.0, im = 0.0;
    for (int i = lane; i < g.Nx; i += 32) {
        const cplx<T> v = F.at(row, i);
        const double2 w = wx[PSATD_IX(i, g.Nx)];
        re += w.x * (double)v.x - w.y * (double)v.y;
        im += w.x * (double)v.y + w.y * (double)v.x;
    }
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, o);
        im += __shfl_down_sync(0xffffffffu, im, o);
    }
    if (lane == 0) out[PSATD_IX(warp, rows)] = make_double2(re, im);
}

// h[a][l][p] = sum_j wy[p][j] g[a][l][j]
__global__ void contract_y_kernel(const double2* __restrict__ gin, GridGeom g, int ncomp, int ny,
                                  const double2* __restrict__ wy, double2* __restrict__ h) {
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (tid >= (long long)ncomp * g.Nz * ny) return;
    const int p = (int)(tid % ny);
    const long long al = tid / ny;                 // a * Nz + l
    const double2* gr = gin + (size_t)al * g.Ny;
    const double2* w = wy + (size_t)p * g.Ny;
    double re = 0.0, im = 0.0;
    const GBuf<const double2> Gi{gin, (long long)ncomp * g.Nz * g.Ny}, Wy{wy, (long long)ny * g.Ny};
    for (int j = 0; j < g.Ny; ++j) {
        const double2 a = Gi.at(gr, j), b = Wy.at(w, j);
        re += b.x * a.x - b.y * a.y;
        im += b.x * a.y + b.y * a.x;
    }
    h[PSATD_IX(tid, (long long)ncomp * g.Nz * ny)] = make_double2(re, im);
}

// out[a][q][p] = I_S(x_p, y_p, z_q, t) * sum_l wz[q][l] h[a][l][p]
template <typename T>
__global__ void contract_z_kernel(const double2* __restrict__ h, GridGeom g, ShellGeom sh, int ncomp,
                                  int ny, int nz, double x_phys, double y0, double y1, double z0,
                                  double z1, double t, const double2* __restrict__ wz,
                                  cplx<T>* __restrict__ out) {
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (tid >= (long long)ncomp * nz * ny) return;
    const int p = (int)(tid % ny);
    const long long r = tid / ny;
    const int q = (int)(r % nz);
    const int a = (int)(r / nz);
    const double2* w = wz + (size_t)q * g.Nz;
    const double2* hc = h + (size_t)a * g.Nz * ny + p;
    double re = 0.0, im = 0.0;
    const GBuf<const double2> Hb{h, (long long)ncomp * g.Nz * ny}, Wz{wz, (long long)nz * g.Nz};
    for (int l = 0; l < g.Nz; ++l) {
        const double2 v = Hb.at(hc, (long long)l * ny), b = Wz.at(w, l);
        re += b.x * v.x - b.y * v.y;
        im += b.x * v.y + b.y * v.x;
    }
    const double y = y0 + (y1 - y0) * p / ny;
    const double z = z0 + (z1 - z0) * q / nz;
    const double m = cut_out_indicator(x_phys, y, z, t, sh, g.c);
    out[PSATD_IX(tid, (long long)ncomp * nz * ny)] = mk<T>((T)(re * m), (T)(im * m));
}

// ---------------------------------------------------------------------------
// float32 storage: the same three contractions in double-float arithmetic
// (weights, g and h as float4 double-float complex values; the sums are the
// compensated ones of ff.cuh's Dot2).  All three are bound by the float32 pipe
// (12 or 13 instructions per real product), so each is laid out to keep every
// SM's pipe busy: 8 lanes a row instead of a warp a row along x (3 instead of 5
// rounds of the cross-lane sum), and register tiles with the sum split over the
// warps of a block along y and z.
// With the sums in chains of renormalised pairs, a warp a row and a thread an
// output, the four kernels of a plane of 64 x 64 points and three components on
// a 128^3 layer took 8.5 (weights), 27.5 (x), 31.7 (y) and 75 us (z), and 64 such
// planes with their copies 7.7 ms; now the 64 planes take 2.7 ms, most of it the
// host's calls.  One-shot of a 256^3 real box with a plane of 128 x 128: 1.22 ->
// 0.94 ms.

constexpr int kXL = 8;                          // lanes per row of the x contraction
constexpr int kXLFew = 32;                      // ... where there are few rows
constexpr int kXThreads = 256;

// sum over the XL lanes of a row's group (every lane gets the total)
template <int XL = kXL>
__device__ __forceinline__ CFF group_sum(CFF a) {
#pragma unroll
    for (int o = XL / 2; o > 0; o >>= 1) {
        CFF b;
        b.re.h = __shfl_xor_sync(0xffffffffu, a.re.h, o);
        b.re.l = __shfl_xor_sync(0xffffffffu, a.re.l, o);
        b.im.h = __shfl_xor_sync(0xffffffffu, a.im.h, o);
        b.im.l = __shfl_xor_sync(0xffffffffu, a.im.l, o);
        a = cff_add(a, b);
    }
    return a;
}

// g[a][l][j] = sum_i wx[i] f[c_a][l][j][i]; XL lanes take kXRows rows (a, l, j)
// half the rows apart, whose loads are in flight together and share each weight.
// REAL: f holds float32 values (Nx even), else complex float32 ones.
constexpr int kXRows = 2;
template <bool REAL, int XL, int BLOCKS>
__global__ void __launch_bounds__(kXThreads, BLOCKS)
contract_x_ff_kernel(const float* __restrict__ f, GridGeom g, CompList cl, int ncomp,
                     const float4* __restrict__ wx, float4* __restrict__ out) {
    extern __shared__ float4 sw[];                            // the weights, [Nx]
    pdl_launch_dependents();
    pdl_wait();
    for (int i = threadIdx.x; i < g.Nx; i += kXThreads) sw[i] = wx[PSATD_IX(i, g.Nx)];
    __syncthreads();
    const int lane = threadIdx.x % XL;
    const long long per_comp = (long long)g.Nz * g.Ny, rows = ncomp * per_comp;
    const long long units = (rows + kXRows - 1) / kXRows;
    const long long unit = blockIdx.x * (long long)(kXThreads / XL) + threadIdx.x / XL;
    long long row[kXRows];
    bool have[kXRows];                                        // (every lane takes part in the sums)
    const float2* p[kXRows];
    const float2* f2 = reinterpret_cast<const float2*>(f);
    const int n2 = REAL ? g.Nx / 2 : g.Nx;                    // float2 per row
#pragma unroll
    for (int r = 0; r < kXRows; ++r) {
        row[r] = unit + r * units;
        have[r] = unit < units && row[r] < rows;
        const long long r0 = have[r] ? row[r] : 0;
        const int a = (int)(r0 / per_comp);
        p[r] = f2 + ((size_t)cl.c[a] * per_comp + (size_t)(r0 - a * per_comp)) * n2;
    }
    const GBuf<const float2> F{f2, 6LL * per_comp * n2};
    Dot2C acc[kXRows] = {};
    auto mac = [&](int r, int i, float2 v) {
        if constexpr (REAL) dot2_mac_real(acc[r], sw[2 * i], sw[2 * i + 1], v);
        else dot2_mac(acc[r], sw[i], v);
    };
    int i = lane;
#pragma unroll 1
    for (; i + 3 * XL < n2; i += 4 * XL) {
        float2 v[kXRows][4];                                  // (all eight loads before the sums)
#pragma unroll
        for (int e = 0; e < 4 * kXRows; ++e) v[e / 4][e % 4] = F.at(p[e / 4], i + e % 4 * XL);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int r = 0; r < kXRows; ++r) {
                mac(r, i + k * XL, v[r][k]);
                if (k % 2) dot2_norm(acc[r]);
            }
    }
    for (; i < n2; i += XL)
#pragma unroll
        for (int r = 0; r < kXRows; ++r) {
            mac(r, i, F.at(p[r], i));
            dot2_norm(acc[r]);
        }
#pragma unroll
    for (int r = 0; r < kXRows; ++r) {
        const CFF t = group_sum<XL>(dot2_value(acc[r]));
        if (have[r] && lane == 0) out[PSATD_IX(row[r], rows)] = cff_store(t);
    }
}

// XL lanes a row: 8 (fewer rounds of the cross-lane sum) unless that leaves the SMs
// without two blocks each and a row is long enough for 32.  Three components of 64 x 64
// points on 1000 x 64 x 64 118 -> 48 us, on 2048 x 32 x 32 127 -> 44 us (104 and 64 us
// with a warp a row in renormalised sums); 32 lanes everywhere make the 256^3 real plane
// of 128 x 128 points 167 -> 196 us.
// Five blocks an SM (48 registers) keep a row's loads in flight together (256 x 128 x
// 128, three components 63 -> 51 us against six).  A grid of short rows that fits six an
// SM but not five takes six, without a second wave of a few blocks (128^3, three
// components 46 -> 38 us; complex fields: real ones, 256 points a row, would spill).
template <bool REAL>
cudaError_t contract_x_ff(const float* f, const GridGeom& g, const CompList& cl, int ncomp, const float4* wx,
                          float4* out, cudaStream_t s) {
    const long long units = ((long long)ncomp * g.Nz * g.Ny + kXRows - 1) / kXRows;
    auto launch = [&](auto lanes, auto blocks) {
        constexpr int XL = decltype(lanes)::value, per = kXThreads / XL;
        return launch_pdl(contract_x_ff_kernel<REAL, XL, decltype(blocks)::value>,
                          dim3((unsigned)((units + per - 1) / per)), kXThreads, (size_t)g.Nx * sizeof(float4), s, f, g,
                          cl, ncomp, wx, out);
    };
    using Five = std::integral_constant<int, 5>;
    using Six = std::integral_constant<int, 6>;
    const long long blocks = (units * kXL + kXThreads - 1) / kXThreads;
    if (blocks < 2 * 152 && g.Nx >= 128) return launch(std::integral_constant<int, kXLFew>{}, Five{});
    if constexpr (!REAL)
        if (blocks > 5 * 152 && blocks <= 6 * 152 && g.Nx < 192) return launch(std::integral_constant<int, kXL>{}, Six{});
    return launch(std::integral_constant<int, kXL>{}, Five{});
}

// Half spectrum of real fields (slots p < Nx/2 holding x mode mode[p], the x
// Nyquist mode in Q), with the 1/N of the inverse DFT folded in.  The modes with
// negative k_x are the conjugates F(-k) = conj F(k) of the stored ones, so with
//   A  = sum_{p: mode 1..Nx/2-1} S[p] wx[mode[p]],   Z = S[0] wx[0] + Q wx[Nx/2]
// of a row (l, j) and those of its mirror row (-l, -j) (indices mod N),
//   g[l][j] = Z[l][j] + A[l][j] + conj(A[-l][-j]),
// using conj(F) wx[-k_x] = conj(F wx[k_x]).  kXL lanes take a row and its mirror
// and write both, so each row is read and summed once: l = 0 .. Nz/2, and the
// pairs of l = 0 and l = Nz/2 only once (j <= their mirror).
__global__ void __launch_bounds__(kXThreads, 5)
contract_x_half_ff_kernel(const float2* __restrict__ S, const float2* __restrict__ Q, GridGeom g, CompList cl,
                          int ncomp, const int* __restrict__ mode, const float4* __restrict__ wx,
                          float4* __restrict__ out) {
    extern __shared__ float4 sw[];                            // the weights in slot order, then wx[Nx/2]
    pdl_launch_dependents();
    pdl_wait();
    const int nh = g.Nx / 2;
    for (int i = threadIdx.x; i <= nh; i += kXThreads)
        sw[i] = wx[PSATD_IX(i == nh ? nh : mode[PSATD_IX(i, nh)], g.Nx)];
    __syncthreads();
    const int lane = threadIdx.x % kXL;
    const int hz = g.Nz / 2 + 1;
    const long long units = (long long)ncomp * hz * g.Ny;
    const long long u = blockIdx.x * (long long)(kXThreads / kXL) + threadIdx.x / kXL;
    const long long u0 = u < units ? u : 0;
    const int a = (int)(u0 / ((long long)hz * g.Ny));
    const int l = (int)(u0 / g.Ny % hz), j = (int)(u0 % g.Ny);
    const int lm = (g.Nz - l) % g.Nz, jm = (g.Ny - j) % g.Ny;
    const bool have = u < units && (lm != l || j <= jm);
    const size_t cbase = (size_t)cl.c[a] * g.Nz * g.Ny;
    const size_t ra = cbase + (size_t)l * g.Ny + j, rm = cbase + (size_t)lm * g.Ny + jm;
    const float2 *pa = S + ra * nh, *pm = S + rm * nh;
    const GBuf<const float2> SF{S, 6LL * g.Nz * g.Ny * nh};
    Dot2C A{}, Am{};
    if (have) {
        // slot 0 holds x mode 0: its term belongs to Z
        int p = lane ? lane : kXL;
#pragma unroll 1
        for (; p + 3 * kXL < nh; p += 4 * kXL) {
            float2 v[4], vm[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v[k] = SF.at(pa, p + k * kXL);
                vm[k] = SF.at(pm, p + k * kXL);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                dot2_mac(A, sw[p + k * kXL], v[k]);
                dot2_mac(Am, sw[p + k * kXL], vm[k]);
                if (k % 2) {
                    dot2_norm(A);
                    dot2_norm(Am);
                }
            }
        }
        for (; p < nh; p += kXL) {
            dot2_mac(A, sw[p], SF.at(pa, p));
            dot2_mac(Am, sw[p], SF.at(pm, p));
            dot2_norm(A);
            dot2_norm(Am);
        }
    }
    const CFF sa = group_sum(dot2_value(A)), sm = group_sum(dot2_value(Am));
    if (have && lane < 2) {                                   // lane 0 writes the row, lane 1 its mirror
        const CFF own = lane ? sm : sa, oth = lane ? sa : sm;
        const size_t r = lane ? rm : ra;
        Dot2C Z{};
        dot2_mac(Z, sw[0], SF.at(lane ? pm : pa, 0));
        dot2_mac(Z, sw[nh], Q[PSATD_IX(r, 6LL * g.Nz * g.Ny)]);
        const CFF z = dot2_value(Z);
        const CFF t{ff_add(z.re, ff_add(own.re, oth.re)), ff_add(z.im, ff_sub(own.im, oth.im))};
        out[PSATD_IX((size_t)a * g.Nz * g.Ny + (r - cbase), (long long)ncomp * g.Nz * g.Ny)] = cff_store(t);
    }
}

// The y and z contractions as double-float complex products C[m][n] = sum_k
// A[m][k] B[k][n].  A block takes a tile of 8 R x 8 R outputs (R x R a thread;
// R = 2: four products per four 16-byte shared loads) and splits k over kCS groups
// of 64 threads, whose sums are added in a fixed order at the end: without the
// split the smallest planes leave a warp or two per SM.  R = 2 when it still gives
// every SM two tiles, else R = 1 (four times the tiles; the float32 pipe stays the
// bound, 51 instructions per product against two shared loads).  Operands come in chunks of 32 k
// through shared memory, the next chunk loaded while one is multiplied; rows are
// 33 float4 apart, so the eight rows a quarter-warp reads lie on distinct banks.
//   y: m = (a, l), k = j, n = p:  A = g, B[k][n] = wy[n][k];
//   z: m = q, k = l, n = p, one a per blockIdx.z:  A = wz, B = h; the result times
//      the cut-out, rounded to float32.
constexpr int kCK = 32, kCS = 4, kCThreads = 64 * kCS, kCRow = kCK + 1;

template <bool ZAX, int R>
__global__ void __launch_bounds__(kCThreads)
contract_yz_ff_kernel(const float4* __restrict__ A, const float4* __restrict__ B, int M, int N, int K,
                      float4* __restrict__ h, GridGeom g, ShellGeom sh, double x_phys, double y0, double y1, double z0,
                      double z1, double t, float2* __restrict__ out) {
    constexpr int kCT = 8 * R;
    __shared__ float4 sA[kCT * kCRow], sB[kCT * kCRow];
    __shared__ float4 part[kCS - 1][R * R][64];
    pdl_launch_dependents();
    pdl_wait();
    const int tid = threadIdx.x, grp = tid / 64, tx = tid % 8, ty = (tid % 64) / 8;
    const int m0 = blockIdx.y * kCT, n0 = blockIdx.x * kCT, a = blockIdx.z;
    const float4* Bp = ZAX ? B + (size_t)a * K * N : B;
    const GBuf<const float4> GA{A, (long long)M * K}, GB{B, (long long)gridDim.z * K * N};
    constexpr int PER = kCT * kCK / kCThreads;                // float4 of one operand per thread and chunk
    float4 ra[PER], rb[PER];
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int e = tid + i * kCThreads;
            const int r = e / kCK, k = k0 + e % kCK;
            ra[i] = (m0 + r < M && k < K) ? GA.at(A, (long long)(m0 + r) * K + k) : zero;
            if constexpr (ZAX) {
                const int kk = k0 + e / kCT, n = n0 + e % kCT;       // 16 consecutive n of one k
                rb[i] = (n < N && kk < K) ? GB.at(Bp, (long long)kk * N + n) : zero;
            } else {
                rb[i] = (n0 + r < N && k < K) ? GB.at(Bp, (long long)(n0 + r) * K + k) : zero;
            }
        }
    };
    Dot2C acc[R][R] = {};
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += kCK) {
        __syncthreads();                                      // the last chunk has been read
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int e = tid + i * kCThreads;
            sA[(e / kCK) * kCRow + e % kCK] = ra[i];
            if constexpr (ZAX) sB[(e % kCT) * kCRow + e / kCT] = rb[i];
            else sB[(e / kCK) * kCRow + e % kCK] = rb[i];
        }
        __syncthreads();
        if (k0 + kCK < K) fetch(k0 + kCK);
#pragma unroll 1
        for (int kb = grp; kb < kCK; kb += 2 * kCS) {
#pragma unroll
            for (int k = kb; k < kb + 2 * kCS; k += kCS) {
                float4 av[R], bv[R];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    av[i] = sA[(ty + 8 * i) * kCRow + k];
                    bv[i] = sB[(tx + 8 * i) * kCRow + k];
                }
#pragma unroll
                for (int i = 0; i < R * R; ++i) dot2_mac_cff(acc[i / R][i % R], av[i / R], bv[i % R]);
            }
#pragma unroll
            for (int i = 0; i < R * R; ++i) dot2_norm(acc[i / R][i % R]);
        }
    }
    if (grp > 0) {
#pragma unroll
        for (int i = 0; i < R * R; ++i) part[grp - 1][i][tid % 64] = cff_store(dot2_value(acc[i / R][i % R]));
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int i = 0; i < R * R; ++i) {
        CFF v = dot2_value(acc[i / R][i % R]);
#pragma unroll
        for (int s = 0; s < kCS - 1; ++s) v = cff_add(v, cff_load(part[s][i][tid]));
        const int m = m0 + ty + 8 * (i / R), n = n0 + tx + 8 * (i % R);
        if (m >= M || n >= N) continue;
        if constexpr (ZAX) {
            const float w = cut_out_f(x_phys, y0, y1, n, N, z0, z1, m, M, t, sh, g.c);
            out[PSATD_IX(((size_t)a * M + m) * N + n, (long long)gridDim.z * M * N)] =
                make_float2(ff_float(v.re) * w, ff_float(v.im) * w);
        } else {
            h[PSATD_IX((size_t)m * N + n, (long long)M * N)] = cff_store(v);
        }
    }
}

// y and z contractions of float32 storage (g and the weights are in the scratch)
cudaError_t contract_yz_ff(const GridGeom& g, const ShellGeom& sh, double x_phys, int ny, int nz, double y0, double y1,
                           double z0, double z1, double t, int ncomp, const SampleScratch& sc, float2* out,
                           cudaStream_t s) {
    const float4 *gg = reinterpret_cast<const float4*>(sc.g), *wy = reinterpret_cast<const float4*>(sc.wy);
    const float4 *hh = reinterpret_cast<const float4*>(sc.h), *wz = reinterpret_cast<const float4*>(sc.wz);
    const int rows = ncomp * g.Nz;
    auto launch = [&](auto zax, auto rc) {
        constexpr bool Z = decltype(zax)::value;
        constexpr int R = decltype(rc)::value;
        auto tiles = [](int n) { return (unsigned)((n + 8 * R - 1) / (8 * R)); };
        if constexpr (Z)
            return launch_pdl(contract_yz_ff_kernel<true, R>, dim3(tiles(ny), tiles(nz), (unsigned)ncomp), kCThreads,
                                0, s, wz, hh, nz, ny, g.Nz, (float4*)nullptr, g, sh, x_phys, y0, y1, z0, z1, t, out);
        else
            return launch_pdl(contract_yz_ff_kernel<false, R>, dim3(tiles(ny), tiles(rows), 1), kCThreads, 0, s, gg,
                                wy, rows, ny, g.Ny, reinterpret_cast<float4*>(sc.h), g, sh, x_phys, y0, y1, z0, z1, t,
                                (float2*)nullptr);
    };
    auto wide = [&](long long m) { return ((m + 15) / 16) * ((ny + 15) / 16) >= 2 * 152; };
    using One = std::integral_constant<int, 1>;
    using Two = std::integral_constant<int, 2>;
    cudaError_t e = wide(rows) ? launch(std::false_type{}, Two{}) : launch(std::false_type{}, One{});
    if (e != cudaSuccess) return e;
    return wide((long long)nz * ncomp) ? launch(std::true_type{}, Two{}) : launch(std::true_type{}, One{});
}

}  // namespace

template <typename T>
cudaError_t launch_sample_plane(const cplx<T>* data, const GridGeom& g, const ShellGeom& sh,
                                double x_phys, int ny, int nz, double y0, double y1, double z0,
                                double z1, double t, const int* comps, int ncomp,
                                const SampleScratch& sc, cplx<T>* out, cudaStream_t s,
                                long long* nlaunch, bool from_spectrum) {
    CompList cl;
    for (int a = 0; a < 6; ++a) cl.c[a] = a < ncomp ? comps[a] : 0;
    const int nw = g.Nx + ny * g.Ny + nz * g.Nz;
    const dim3 wgrid((nw + kWThreads - 1) / kWThreads);
    cudaError_t e;
    constexpr bool ffw = sizeof(T) == 4;               // float32 storage: double-float sums
    if (from_spectrum)
        e = launch_pdl(spectral_weights_kernel<ffw>, wgrid, kWThreads, 0, s, g, x_phys, ny, nz, y0, y1, z0, z1, sc.wx, sc.wy,
                         sc.wz);
    else
        e = launch_pdl(weights_kernel<ffw>, wgrid, kWThreads, 0, s, g, x_phys, ny, nz, y0, y1, z0, z1, sc.wx, sc.wy,
                         sc.wz);
    if constexpr (ffw) {
        if (e != cudaSuccess) return e;
        e = contract_x_ff<false>(reinterpret_cast<const float*>(data), g, cl, ncomp,
                                 reinterpret_cast<const float4*>(sc.wx), reinterpret_cast<float4*>(sc.g), s);
        if (e == cudaSuccess)
            e = contract_yz_ff(g, sh, x_phys, ny, nz, y0, y1, z0, z1, t, ncomp, sc, reinterpret_cast<float2*>(out), s);
        if (nlaunch) *nlaunch += 4;
        return e;
    } else {
        if (e != cudaSuccess) return e;
        const long long rows = (long long)ncomp * g.Nz * g.Ny;
        const long long nh = (long long)ncomp * g.Nz * ny;
        const long long no = (long long)ncomp * nz * ny;
        contract_x_kernel<T><<<(unsigned)((rows * 32 + 255) / 256), 256, 0, s>>>(data, g, cl, ncomp, sc.wx, sc.g);
        contract_y_kernel<<<(unsigned)((nh + 255) / 256), 256, 0, s>>>(sc.g, g, ncomp, ny, sc.wy, sc.h);
        contract_z_kernel<T><<<(unsigned)((no + 255) / 256), 256, 0, s>>>(sc.h, g, sh, ncomp, ny, nz, x_phys,
                                                                          y0, y1, z0, z1, t, sc.wz, out);
        if (nlaunch) *nlaunch += 4;
        return cudaGetLastError();
    }
}

cudaError_t launch_sample_plane_real(const float* data, const float2* nyq, const int* slot_mode, const GridGeom& g,
                                     const ShellGeom& sh, double x_phys, int ny, int nz, double y0, double y1,
                                     double z0, double z1, double t, const int* comps, int ncomp,
                                     const SampleScratch& sc, float2* out, cudaStream_t s, long long* nlaunch,
                                     bool from_spectrum) {
    CompList cl;
    for (int a = 0; a < 6; ++a) cl.c[a] = a < ncomp ? comps[a] : 0;
    const int nw = g.Nx + ny * g.Ny + nz * g.Nz;
    const dim3 wgrid((nw + kWThreads - 1) / kWThreads);
    cudaError_t e;
    if (from_spectrum)
        e = launch_pdl(spectral_weights_kernel<true>, wgrid, kWThreads, 0, s, g, x_phys, ny, nz, y0, y1, z0, z1, sc.wx, sc.wy,
                         sc.wz);
    else
        e = launch_pdl(weights_kernel<true>, wgrid, kWThreads, 0, s, g, x_phys, ny, nz, y0, y1, z0, z1, sc.wx, sc.wy,
                         sc.wz);
    const float4* wx = reinterpret_cast<const float4*>(sc.wx);
    float4* gg = reinterpret_cast<float4*>(sc.g);
    if (e != cudaSuccess) return e;
    constexpr int per = kXThreads / kXL;
    if (from_spectrum) {
        const long long units = (long long)ncomp * (g.Nz / 2 + 1) * g.Ny;
        e = launch_pdl(contract_x_half_ff_kernel, dim3((unsigned)((units + per - 1) / per)), kXThreads,
                         (size_t)(g.Nx / 2 + 1) * sizeof(float4), s, reinterpret_cast<const float2*>(data), nyq, g, cl,
                         ncomp, slot_mode, wx, gg);
    } else {
        e = contract_x_ff<true>(data, g, cl, ncomp, wx, gg, s);
    }
    if (e == cudaSuccess) e = contract_yz_ff(g, sh, x_phys, ny, nz, y0, y1, z0, z1, t, ncomp, sc, out, s);
    if (nlaunch) *nlaunch += 4;
    return e;
}

template cudaError_t launch_sample_plane<float>(const cplx<float>*, const GridGeom&, const ShellGeom&, double, int, int, double, double, double, double, double, const int*, int, const SampleScratch&, cplx<float>*, cudaStream_t, long long*, bool);
template cudaError_t launch_sample_plane<double>(const cplx<double>*, const GridGeom&, const ShellGeom&, double, int, int, double, double, double, double, double, const int*, int, const SampleScratch&, cplx<double>*, cudaStream_t, long long*, bool);

}  // namespace psatd
