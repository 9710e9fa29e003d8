// float32 y and z transforms of 512 = 8 x 8 x 8 and 1024 = 16 x 8 x 8 points: the
// in-place passes of fft_mixed.cuh with the radices, the tile and every shared-memory
// offset fixed at compile time.
//
// A block takes 16 x-columns (128 bytes a row: at 1024^2 planes narrower rows use the
// DRAM bursts poorly), the tile in shared memory once (64 or 128 KB).  Bound by memory
// traffic, one read and one write, if enough of it is in flight: three passes of at
// most 16 points need 64 registers a thread, so 1024 threads share an SM, against 512
// at 128 registers for the two passes of 32 points of fft_fast.cu, whose loads,
// transforms and stores barely overlapped.  One more pass through shared memory costs
// less than the warps gain.  Per launch, two passes of 32 x 16 (32 x 32) points
// against this: 512^3 y 2.78 -> 2.49 ms, z 3.16 -> 2.55 ms (5.05 TB/s); 1024 x 1024 x
// 512 y 11.9 -> 11.6 ms.
#include "fft_mixed.cuh"

namespace psatd {

namespace {

constexpr int kW = 16;

template <int R1, int R2, int R3, int TH, int S>
__global__ void __launch_bounds__(TH, 1024 / TH)
three_cols_kernel(float2* __restrict__ data, int axis, int Nx, int Ny, int Nz, int ncomp,
                  const float2* __restrict__ tp) {
    constexpr int N = R1 * R2 * R3, L1 = N / R1, L2 = L1 / R2;          // runs of the first and second level
    static_assert(L2 == R3, "three levels");
    extern __shared__ __align__(16) unsigned char three_smem[];
    float2* sm = reinterpret_cast<float2*>(three_smem);                // [N][kW]
    const unsigned ntile = (unsigned)(Nx + kW - 1) / kW, outer = axis == 1 ? Nz : Ny;
    const unsigned rest = blockIdx.x / ntile, x0 = (blockIdx.x - rest * ntile) * kW;
    const unsigned comp = rest / outer, o = rest - comp * outer;
    const size_t plane = (size_t)Nx * Ny, stride = axis == 1 ? (size_t)Nx : plane;
    const int c = threadIdx.x % kW, t0 = threadIdx.x / kW;
    constexpr int U = TH / kW;                                          // items of a column at a time
    float2* base = data + comp * plane * Nz + (axis == 1 ? o * plane : (size_t)o * Nx) + x0 + c;
    const GBuf<float2> F{data, (long long)ncomp * plane * Nz};
    const bool col = x0 + c < (unsigned)Nx;
    pdl_launch_dependents();
    pdl_wait();
    if (col) {
#pragma unroll
        for (int n = 0; n < L1 / U; ++n) {
            const int j = t0 + n * U;
            float2 v[R1];
            const float2* p = base + j * stride;
            static_for<0, R1>([&](auto rc) {
                v[decltype(rc)::value] = F.at(p, 0);
                p += L1 * stride;
            });
            reg_dft<float, S, R1>(v);
            static_for<1, R1>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const float2 w = tp[PSATD_IX(k * L1 + j, 2 * N)];
                v[k] = S < 0 ? cmul(v[k], w) : cmulc(v[k], w);
            });
            static_for<0, R1>([&](auto kc) { sm[(decltype(kc)::value * L1 + j) * kW + c] = v[decltype(kc)::value]; });
        }
    }
    __syncthreads();
    if (col) {
#pragma unroll
        for (int n = 0; n < N / R2 / U; ++n) {
            const int u = t0 + n * U, blk = u / L2, j = u - blk * L2;
            float2* s = sm + (blk * L1 + j) * kW + c;
            float2 v[R2];
            static_for<0, R2>([&](auto rc) { v[decltype(rc)::value] = s[decltype(rc)::value * L2 * kW]; });
            reg_dft<float, S, R2>(v);
            static_for<1, R2>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const float2 w = tp[PSATD_IX(N + k * L2 + j, 2 * N)];
                v[k] = S < 0 ? cmul(v[k], w) : cmulc(v[k], w);
            });
            static_for<0, R2>([&](auto rc) { s[decltype(rc)::value * L2 * kW] = v[decltype(rc)::value]; });
        }
    }
    __syncthreads();
    if (col) {
#pragma unroll
        for (int n = 0; n < N / R3 / U; ++n) {
            const int u = t0 + n * U;                                    // u = k1 R2 + k2
            const float2* s = sm + u * R3 * kW + c;
            float2 v[R3];
            static_for<0, R3>([&](auto rc) { v[decltype(rc)::value] = s[decltype(rc)::value * kW]; });
            reg_dft<float, S, R3>(v);
            const int k1 = u / R2, k2 = u - k1 * R2;
            float2* p = base + (size_t)(k1 + R1 * k2) * stride;
            static_for<0, R3>([&](auto rc) {
                F.at(p, 0) = v[decltype(rc)::value];
                p += (size_t)(R1 * R2) * stride;
            });
        }
    }
}

template <int R1, int R2, int R3, int TH>
cudaError_t three_launch(float2* data, int ncomp, const GridGeom& g, const float2* tp, int axis, int dir,
                         cudaStream_t s) {
    const size_t smem = (size_t)R1 * R2 * R3 * kW * sizeof(float2);
    auto k = dir < 0 ? three_cols_kernel<R1, R2, R3, TH, -1> : three_cols_kernel<R1, R2, R3, TH, +1>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long blocks = (long long)ncomp * (axis == 1 ? g.Nz : g.Ny) * ((g.Nx + kW - 1) / kW);
    if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
    return launch_pdl(k, dim3((unsigned)blocks), dim3(TH), smem, s, data, axis, g.Nx, g.Ny, g.Nz, ncomp, tp);
}

}  // namespace

// The y or z transform of a float32 axis of 512 or 1024 points, tp the narrow plan's
// position-ordered twiddles; cudaErrorNotSupported (nothing launched) otherwise.
cudaError_t launch_fft_three(float2* data, int ncomp, const GridGeom& g, const float2* tp, int axis, int dir,
                             cudaStream_t s) {
    const int N = axis == 1 ? g.Ny : g.Nz;
    if (axis == 0) return cudaErrorNotSupported;
    if (N == 512) return three_launch<8, 8, 8, 512>(data, ncomp, g, tp, axis, dir, s);
    if (N == 1024) return three_launch<16, 8, 8, 1024>(data, ncomp, g, tp, axis, dir, s);
    return cudaErrorNotSupported;
}

}  // namespace psatd
