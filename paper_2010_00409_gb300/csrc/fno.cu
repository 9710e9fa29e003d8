// Fourier-neural-operator surrogate: pulse parameters -> focal-region field.
//
// Network (per sample, patch P^3, width C):
//   v0 = W_lift [params, x, y, z] + b_lift                     (pointwise)
//   v_l = act( S_l(v_{l-1}) + W_l v_{l-1} + b_l ),  l = 1..L     (act = GELU, none on l = L)
//   out = W_q2 GELU(W_q1 v_L + b_q1) + b_q2
// S_l is the spectral convolution: truncated DFT of each channel to kx in
// [0, m) (half spectrum, real input) and ky, kz in {0..m-1, P-m..P-1}, a complex
// C x C matrix per kept mode, and the inverse (real output, kx > 0 counted twice).
//
// Every dense contraction is a call of the tensor-core GEMM (gemm.cu): the
// truncated DFTs contract the last axis of their input and write the new
// spectral axis first, so each stage is one strided GEMM per real/imaginary
// part.  All stages are real-linear in the stored (re, im) arrays, so each
// backward stage is the same GEMM with the transposed real matrix.  The
// per-mode complex mixing, GELU, the bias sums, the MSE loss and Adam are small
// elementwise / reduction kernels.  Tensors are float32; GEMM tiles are rounded
// to bfloat16 (float32 accumulation).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <random>
#include <string>
#include <utility>
#include <vector>

#include <cuda_bf16.h>

#include "../../include/psatd.h"
#include "common.cuh"
#include "ff.cuh"

namespace psatd {

namespace {

constexpr double kPi = 3.14159265358979323846;

// ------------------------------------------------------------ small kernels
__global__ void features_kernel(const float* __restrict__ prm, int np, int B, int P, float* __restrict__ feat) {
    const long long nv = (long long)P * P * P;
    const int nch = np + 3;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)B * nch * nv;
         e += (long long)gridDim.x * blockDim.x) {
        const long long vox = e % nv;
        const int ch = (int)((e / nv) % nch);
        const int b = (int)(e / (nv * nch));
        float v;
        if (ch < np) v = prm[b * np + ch];
        else {
            const int x = (int)(vox % P), y = (int)((vox / P) % P), z = (int)(vox / ((long long)P * P));
            const int q = ch == np ? x : (ch == np + 1 ? y : z);
            v = -1.f + 2.f * q / P;
        }
        feat[e] = v;
    }
}

__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// ------------------------------------------------------------ reductions
// Sums over voxels run in three float32 parts up to a warp's sum (72 bits: no less than
// the 53 of a float64 sum of every element, which is bound by the float64 pipe, 1/64 of
// the float32 rate, and took 2.1 ms for 67 M gradients, one block a channel) and in
// float64 from there on.  Rows are cut into kRowChunks pieces so that every SM takes part.
constexpr int kRowChunks = 32;

// SumK with K = 3 of Ogita, Rump and Oishi, "Accurate sum and dot product", 2005: a
// takes the values, b the exact rounding errors of a, c those of b.
struct Sum3 {
    float a, b, c;
};
__device__ __forceinline__ void sum3_add(Sum3& s, float x) {
    const FF t = two_sum(s.a, x), u = two_sum(s.b, t.l);
    s.a = t.h;
    s.b = u.h;
    s.c += u.l;
}

// s, t -> the sum of both
__device__ __forceinline__ Sum3 sum3_merge(const Sum3& s, const Sum3& t) {
    const FF a = two_sum(s.a, t.a), b = two_sum(s.b, t.b), d = two_sum(b.h, a.l);
    return {a.h, d.h, (s.c + t.c) + (b.l + d.l)};
}

// Block sum of one Sum3 per thread (256 threads); thread 0 returns it.
__device__ __forceinline__ double block_sum(Sum3 s) {
    __shared__ Sum3 sh[8];
    for (int o = 16; o > 0; o >>= 1)
        s = sum3_merge(s, Sum3{__shfl_down_sync(0xffffffffu, s.a, o), __shfl_down_sync(0xffffffffu, s.b, o),
                               __shfl_down_sync(0xffffffffu, s.c, o)});
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    double v = 0.0;
    if (threadIdx.x < 32) {
        if (threadIdx.x < 8) {
            const Sum3 t = sh[threadIdx.x];
            v = (double)t.a + ((double)t.b + (double)t.c);
        }
        for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    return v;
}

// Block sum of one float64 value per thread; thread 0 returns it.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double sh[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sh[w];
    return v;
}

// The gradient through an activation and its bias, one read of each operand: with
// GELU gz = ga * gelu'(z), else gz = ga (not written); partial[c][b * kRowChunks +
// chunk] = the sum of the block's gz.  Block (b C + c) kRowChunks + chunk; nv is a multiple of 4.
template <bool GELU>
__global__ void __launch_bounds__(256)
act_back_kernel(const float* __restrict__ z, const float* ga, float* gz, int B, int C,          // gz may be ga
                long long nv, double* __restrict__ partial) {
    const int row = blockIdx.x / kRowChunks, chunk = blockIdx.x % kRowChunks, c = row % C, b = row / C;
    const long long n4 = nv / 4, per = (n4 + kRowChunks - 1) / kRowChunks;
    const long long lo = chunk * per, hi = min(n4, lo + per), off = (long long)row * n4;
    const float4 *z4 = reinterpret_cast<const float4*>(z) + off, *g4 = reinterpret_cast<const float4*>(ga) + off;
    float4* o4 = reinterpret_cast<float4*>(gz) + off;
    Sum3 s{0.f, 0.f, 0.f};
    for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        float4 g = g4[i];
        if constexpr (GELU) {
            const float4 v = z4[i];
            g = make_float4(g.x * gelu_grad(v.x), g.y * gelu_grad(v.y), g.z * gelu_grad(v.z), g.w * gelu_grad(v.w));
            o4[i] = g;
        }
        sum3_add(s, g.x);
        sum3_add(s, g.y);
        sum3_add(s, g.z);
        sum3_add(s, g.w);
    }
    double t;
    if (__syncthreads_or(!isfinite(s.a + s.b + s.c))) {
        // an infinity, a NaN or an overflow, after which the errors are NaN: in float64
        double v = 0.0;
        for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
            const float4 g = GELU ? o4[i] : g4[i];
            v += ((double)g.x + (double)g.y) + ((double)g.z + (double)g.w);
        }
        t = block_sum(v);
    } else {
        t = block_sum(s);
    }
    if (threadIdx.x == 0) partial[(long long)c * B * kRowChunks + b * kRowChunks + chunk] = t;
}

// gbias[c] = the sum of its n partials (one warp a channel, fixed order)
__global__ void bias_reduce_kernel(const double* __restrict__ partial, int n, float* __restrict__ gbias) {
    const double* p = partial + (long long)blockIdx.x * n;
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) s += p[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) gbias[blockIdx.x] = (float)s;
}

// ------------------------------------------------------------ pointwise weight gradients
// gW[o][i] = sum over b, v of gZ[b][o][v] X[b][i][v], operands rounded to bfloat16
// (float32 accumulation): an outer-product reduction over 2 M voxels into 1024
// values, bound by the one read of gZ and X.  A warp walks voxels 16 at a time;
// every operand row is read as float4 (a 16-voxel run is two full sectors a row),
// straight into the fragments of mma.m16n8k16: the four voxels a lane holds are its
// four k slots, the same in both operands, so nothing passes through shared memory.
// (tcgen05 would pad the 32 rows to 128 and stage both operands in shared memory:
// that form took 1.33 ms a layer at 8 x 64^3 voxels, this one 0.09 ms, 6.0 TB/s.)
// Block: 32 x 32 tile (o0, i0) = blockIdx.y, z; splits of the voxels = blockIdx.x.
// Partial tiles go to part[split][Mo][Ni]; wgrad_reduce_kernel adds them in order.
constexpr int kWgWarps = 8;

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__global__ void __launch_bounds__(32 * kWgWarps, 2)
wgrad_kernel(const float* __restrict__ gZ, const float* __restrict__ X, int B, int Mo, int Ni, long long nv,
             float* __restrict__ part) {
    __shared__ float sh[kWgWarps][32][33];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int o0 = blockIdx.y * 32, i0 = blockIdx.z * 32;
    const long long runs = (nv + 15) / 16, total = runs * B;       // 16-voxel runs, batch by batch (nv % 4 == 0)
    const long long nw = (long long)gridDim.x * kWgWarps, w0 = (long long)blockIdx.x * kWgWarps + warp;
    float acc[2][4][4] = {};
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](long long r, float4 (&a)[4], float4 (&x)[4]) {
        const long long b = r / runs, v = (r - b * runs) * 16 + 4 * t;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int o = o0 + 8 * k + g, i = i0 + 8 * k + g;
            a[k] = o < Mo && v < nv ? __ldcs(reinterpret_cast<const float4*>(gZ + (b * Mo + o) * nv + v)) : zero;
            x[k] = i < Ni && v < nv ? __ldcs(reinterpret_cast<const float4*>(X + (b * Ni + i) * nv + v)) : zero;
        }
    };
    float4 a[4], x[4];
    long long r = w0;
    if (r < total) fetch(r, a, x);
    while (r < total) {
        uint32_t af[4][2], xf[4][2];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            af[k][0] = bf16x2(a[k].x, a[k].y); af[k][1] = bf16x2(a[k].z, a[k].w);
            xf[k][0] = bf16x2(x[k].x, x[k].y); xf[k][1] = bf16x2(x[k].z, x[k].w);
        }
        r += nw;
        if (r < total) fetch(r, a, x);
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n = 0; n < 4; ++n)
                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                             "{%0,%1,%2,%3};"
                             : "+f"(acc[m][n][0]), "+f"(acc[m][n][1]), "+f"(acc[m][n][2]), "+f"(acc[m][n][3])
                             : "r"(af[2 * m][0]), "r"(af[2 * m + 1][0]), "r"(af[2 * m][1]), "r"(af[2 * m + 1][1]),
                               "r"(xf[n][0]), "r"(xf[n][1]));
    }
    // c0, c1: row g, columns 2t, 2t + 1; c2, c3: row g + 8
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            sh[warp][16 * m + g][8 * n + 2 * t] = acc[m][n][0];
            sh[warp][16 * m + g][8 * n + 2 * t + 1] = acc[m][n][1];
            sh[warp][16 * m + g + 8][8 * n + 2 * t] = acc[m][n][2];
            sh[warp][16 * m + g + 8][8 * n + 2 * t + 1] = acc[m][n][3];
        }
    __syncthreads();
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
        const int o = e >> 5, i = e & 31;
        if (o0 + o >= Mo || i0 + i >= Ni) continue;
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kWgWarps; ++w) s += sh[w][o][i];
        part[((long long)blockIdx.x * Mo + o0 + o) * Ni + i0 + i] = s;
    }
}

// gW[e] = sum over the splits (a warp an element, float64)
__global__ void wgrad_reduce_kernel(const float* __restrict__ part, int splits, int n, float* __restrict__ gW) {
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (e >= n) return;
    double s = 0.0;
    for (int k = lane; k < splits; k += 32) s += (double)part[(long long)k * n + e];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) gW[e] = (float)s;
}

// ------------------------------------------------------------ per-mode complex mixing
// Spectra laid out [part][mode][b][ch]; weights R[part][mode][i][o].  A block takes
// one mode, its spectra and (backward through the input) its weights in shared
// memory, and a thread four outputs that share each weight, so weights are read from
// memory once and in full lines; bound by the weights' traffic (57 MB a layer at
// 6912 modes and 32 channels).  A thread an output read the weights of the backward
// pass a row apart per lane: 62, 388 and 94 us a layer (forward, input, weights) at a
// batch of 8; now 48, 54 and 47 us.
// A mode's spectra stay in global memory (same layout) where they exceed mix_stage's
// limit.
constexpr int kMixStage = 96 * 1024;

// acc + (x y + z w) in a fixed order of roundings: the product z w, x y added to it in
// one fused operation, the sum.  (Spectra are rounded to bfloat16 by the next
// contraction, so a different order, although no less exact, moves the network's
// output by 4e-5.)
__device__ __forceinline__ float add_dot(float acc, float x, float y, float z, float w) {
    return __fadd_rn(acc, __fmaf_rn(x, y, __fmul_rn(z, w)));
}

// The spectra of one mode, [part][B][C]: staged at sm (stage != 0) or in place.
struct MixSpec { const float *re, *im; };
__device__ __forceinline__ MixSpec mix_spec(const float* g, long long per, int mode, int BC, float* sm, bool stage) {
    const float *re = g + (long long)mode * BC, *im = re + per;
    if (!stage) return {re, im};
    for (int e = threadIdx.x; e < BC; e += blockDim.x) {
        sm[e] = re[e];
        sm[BC + e] = im[e];
    }
    return {sm, sm + BC};
}

// U[mode][b][o] = sum_i V[mode][b][i] R[mode][i][o].  From four samples on a thread
// takes (mode, four b, o), several modes a block when one has few threads' work; the
// modes' spectra are contiguous, so they are staged together.
__global__ void __launch_bounds__(256, 4)
mix_fwd_kernel(const float* __restrict__ V, const float* __restrict__ R, float* __restrict__ U, int modes, int B, int C,
               int per_block, int stage) {
    extern __shared__ float mix_sm[];                              // [2][per_block][B][C]
    constexpr int BT = 4;
    const long long per = (long long)modes * B * C;
    const int mode0 = blockIdx.x * per_block, nm = min(per_block, modes - mode0), BC = B * C;
    const float *vre = V + (long long)mode0 * BC, *vim = vre + per;
    if (stage) {
        for (int e = threadIdx.x; e < nm * BC; e += blockDim.x) {
            mix_sm[e] = vre[e];
            mix_sm[per_block * BC + e] = vim[e];
        }
        vre = mix_sm;
        vim = mix_sm + per_block * BC;
    }
    __syncthreads();
    const int groups = (B + BT - 1) / BT;
    for (int e = threadIdx.x; e < nm * groups * C; e += blockDim.x) {
        const int o = e % C, gm = e / C, m = gm / groups, b0 = (gm - m * groups) * BT, mode = mode0 + m;
        const float* rr = R + (long long)mode * C * C + o;
        const float* ri = rr + (long long)modes * C * C;
        const float *ar = vre + m * BC, *ai = vim + m * BC;
        float ur[BT] = {}, ui[BT] = {};
#pragma unroll 8
        for (int i = 0; i < C; ++i) {
            const float c = rr[i * C], d = ri[i * C];
#pragma unroll
            for (int k = 0; k < BT; ++k) {
                const int bb = min(b0 + k, B - 1);
                const float a = ar[bb * C + i], b = ai[bb * C + i];
                ur[k] = add_dot(ur[k], a, c, -b, d);
                ui[k] = add_dot(ui[k], b, c, a, d);
            }
        }
#pragma unroll
        for (int k = 0; k < BT; ++k)
            if (b0 + k < B) {
                const long long q = ((long long)mode * B + b0 + k) * C + o;
                U[q] = ur[k];
                U[per + q] = ui[k];
            }
    }
}

// The same with a thread an output, for one to three samples (a weight then serves
// at most three outputs: 15 us a layer at one sample against 23 us for the above).
__global__ void mix_fwd_few_kernel(const float* __restrict__ V, const float* __restrict__ R, float* __restrict__ U,
                                   int modes, int B, int C) {
    const long long per = (long long)modes * B * C;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < per; e += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(e % C);
        const long long mb = e / C;                      // mode * B + b
        const int mode = (int)(mb / B);
        const float* vr = V + mb * C;
        const float* vi = V + per + mb * C;
        const float* rr = R + (long long)mode * C * C + o;
        const float* ri = R + (long long)modes * C * C + (long long)mode * C * C + o;
        float ur = 0.f, ui = 0.f;
        for (int i = 0; i < C; ++i) {
            const float a = vr[i], b = vi[i], c = rr[i * C], d = ri[i * C];
            ur = add_dot(ur, a, c, -b, d);
            ui = add_dot(ui, b, c, a, d);
        }
        U[e] = ur;
        U[per + e] = ui;
    }
}

// gV[mode][b][i] = sum_o (gUr R_r + gUi R_i, -gUr R_i + gUi R_r): thread i, four b a
// thread, rows of R a row stride of C + 1 apart in shared memory, `rows` at a time.
__global__ void mix_back_input_kernel(const float* __restrict__ gU, const float* __restrict__ R,
                                      float* __restrict__ gV, int modes, int B, int C, int rows, int stage) {
    extern __shared__ float mix_sm[];                              // [2][B][C] gradients, [2][rows][C + 1] weights
    const long long per = (long long)modes * B * C;
    const int mode = blockIdx.x, BC = B * C, ld = C + 1;
    float *wr = mix_sm + (stage ? 2 * BC : 0), *wi = wr + rows * ld;
    const MixSpec u = mix_spec(gU, per, mode, BC, mix_sm, stage);
    const float* rr = R + (long long)mode * C * C;
    const float* ri = R + (long long)modes * C * C + (long long)mode * C * C;
    const int groups = (B + 3) / 4;
    for (int r0 = 0; r0 < C; r0 += rows) {
        const int nr = min(rows, C - r0);
        __syncthreads();
        for (int e = threadIdx.x; e < nr * C; e += blockDim.x) {
            const int i = e / C, o = e - i * C;
            wr[i * ld + o] = rr[r0 * C + e];
            wi[i * ld + o] = ri[r0 * C + e];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < groups * nr; e += blockDim.x) {
            const int i = e % nr, b0 = (e / nr) * 4;
            float vr[4] = {}, vi[4] = {};
#pragma unroll 4
            for (int o = 0; o < C; ++o) {
                const float c = wr[i * ld + o], d = wi[i * ld + o];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int bb = min(b0 + k, B - 1);
                    const float a = u.re[bb * C + o], b = u.im[bb * C + o];
                    vr[k] = add_dot(vr[k], a, c, b, d);
                    vi[k] = add_dot(vi[k], b, c, -a, d);
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (b0 + k < B) {
                    const long long q = ((long long)mode * B + b0 + k) * C + r0 + i;
                    gV[q] = vr[k];
                    gV[per + q] = vi[k];
                }
        }
    }
}

// gR[mode][i][o] = sum_b (gUr Vr + gUi Vi, -gUr Vi + gUi Vr): thread o, four i a
// thread.
__global__ void mix_back_weight_kernel(const float* __restrict__ gU, const float* __restrict__ V,
                                       float* __restrict__ gR, int modes, int B, int C, int stage) {
    extern __shared__ float mix_sm[];                              // [2][B][C] gradients, [2][B][C] spectra
    const long long per = (long long)modes * B * C, nw = (long long)modes * C * C;
    const int mode = blockIdx.x, BC = B * C;
    const MixSpec u = mix_spec(gU, per, mode, BC, mix_sm, stage);
    const MixSpec v = mix_spec(V, per, mode, BC, mix_sm + 2 * BC, stage);
    __syncthreads();
    float* out = gR + (long long)mode * C * C;
    const int groups = (C + 3) / 4;
    for (int e = threadIdx.x; e < groups * C; e += blockDim.x) {
        const int o = e % C, i0 = (e / C) * 4;
        float sr[4] = {}, si[4] = {};
        for (int b = 0; b < B; ++b) {
            const float gr = u.re[b * C + o], gi = u.im[b * C + o];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = min(i0 + k, C - 1);
                const float vr = v.re[b * C + i], vi = v.im[b * C + i];
                sr[k] = add_dot(sr[k], gr, vr, gi, vi);
                si[k] = add_dot(si[k], gi, vr, -gr, vi);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i0 + k < C) {
                out[(i0 + k) * C + o] = sr[k];
                out[nw + (i0 + k) * C + o] = si[k];
            }
    }
}

// loss partials of mean((y - t)^2) and g = 2 (y - t) / n
__global__ void mse_kernel(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ g, long long n,
                           double* __restrict__ partial) {
    double s = 0.0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const float d = y[e] - t[e];
        s += (double)d * d;
        g[e] = 2.f * d / (float)n;
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            long long n, float lr, float b1, float b2, float eps, float wd, float c1, float c2) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const float gr = g[e] + wd * p[e];
        const float mm = b1 * m[e] + (1.f - b1) * gr;
        const float vv = b2 * v[e] + (1.f - b2) * gr * gr;
        m[e] = mm;
        v[e] = vv;
        p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
}

int grid_for(long long n) {
    long long b = (n + 255) / 256;
    return (int)(b < 152 * 32 ? (b < 1 ? 1 : b) : 152 * 32);
}

}  // namespace

}  // namespace psatd

using namespace psatd;

struct psatd_fno {
    psatd_fno_config cfg{};
    cudaStream_t stream = nullptr;
    int P = 0, C = 0, L = 0, m = 0, NT = 0, MODES = 0, H = 0, NO = 0, NP = 0, maxB = 0;
    long long NV = 0;
    // parameters, gradients, Adam moments (flat)
    float *par = nullptr, *grad = nullptr, *m1 = nullptr, *m2 = nullptr;
    long long npar = 0;
    long long o_lift_w, o_lift_b, o_q1_w, o_q1_b, o_q2_w, o_q2_b;
    std::vector<long long> o_R, o_W, o_b;
    // DFT matrices
    float *Fx = nullptr, *By1 = nullptr, *By2 = nullptr, *Bz1 = nullptr, *Bz2 = nullptr, *Bx1 = nullptr, *Bx2 = nullptr;
    // activations (per layer): input a_l, pre-activation z_l, spectral intermediates
    std::vector<float*> act, pre, T1, T2, T3, U3, W1, W2;
    float *feat = nullptr, *hq = nullptr, *zq = nullptr, *out = nullptr, *gbuf0 = nullptr, *gbuf1 = nullptr;
    float *gT = nullptr, *gT2 = nullptr, *gout = nullptr;
    double *partial = nullptr, *bpart = nullptr;     // loss partials, bias-gradient partials
    float* wpart = nullptr;                          // weight-gradient partials
    int adam_t = 0;
    std::string err = "no error";
};

namespace {

psatd_status fno_fail(psatd_fno* f, psatd_status s, const std::string& m) {
    if (f) f->err = m;
    return s;
}

#define FCK(call)                                                                                 \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) return fno_fail(f, PSATD_ERR_CUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)

// C(m,n) = A(m,k) B(k,n), 1-level batch
GemmArgs G(int M, int N, int K, const float* A, long long sAm, long long sAk, const float* B, long long sBk,
           long long sBn, float* C, long long sCm, long long sCn, float beta, int nb = 1, long long sAb = 0,
           long long sBb = 0, long long sCb = 0) {
    GemmArgs g{};
    g.M = M; g.N = N; g.K = K; g.nb0 = nb; g.nb1 = 1;
    g.A = A; g.sAb0 = sAb; g.sAm = sAm; g.sAk = sAk;
    g.B = B; g.sBb0 = sBb; g.sBk = sBk; g.sBn = sBn;
    g.C = C; g.sCb0 = sCb; g.sCm = sCm; g.sCn = sCn;
    g.alpha = 1.f; g.beta = beta; g.ksplit = 1;
    return g;
}

// Voxel splits of a weight gradient: with its 32 x 32 tiles about two blocks an SM
int wgrad_splits(int Mo, int Ni) {
    const int tiles = ((Mo + 31) / 32) * ((Ni + 31) / 32);
    return std::max(1, 2 * 152 / tiles);
}

int freq_t(int j, int m, int P) { return j < m ? j : P - 2 * m + j; }

}  // namespace

extern "C" {

psatd_status psatd_fno_create(const psatd_fno_config* cfg, unsigned long long seed, void* stream, psatd_fno** out) {
    if (!cfg || !out) return PSATD_ERR_ARG;
    *out = nullptr;
    const int P = cfg->patch, C = cfg->width, L = cfg->layers, m = cfg->modes;
    if (P < 4 || P > 128 || (P & 1) || C < 1 || C > 256 || L < 1 || L > 16 || m < 1 || 2 * m > P ||
        cfg->in_params < 0 || cfg->in_params > 64 || cfg->hidden < 1 || cfg->out_channels < 1 || cfg->max_batch < 1)
        return PSATD_ERR_ARG;
    psatd_fno* f = new (std::nothrow) psatd_fno();
    if (!f) return PSATD_ERR_OOM;
    f->cfg = *cfg;
    f->stream = static_cast<cudaStream_t>(stream);
    f->P = P; f->C = C; f->L = L; f->m = m; f->NT = 2 * m; f->MODES = m * 4 * m * m;
    f->H = cfg->hidden; f->NO = cfg->out_channels; f->NP = cfg->in_params; f->maxB = cfg->max_batch;
    f->NV = (long long)P * P * P;
    const int FI = f->NP + 3;
    // parameter layout
    long long o = 0;
    f->o_lift_w = o; o += (long long)C * FI;
    f->o_lift_b = o; o += C;
    for (int l = 0; l < L; ++l) {
        f->o_R.push_back(o); o += 2LL * f->MODES * C * C;
        f->o_W.push_back(o); o += (long long)C * C;
        f->o_b.push_back(o); o += C;
    }
    f->o_q1_w = o; o += (long long)f->H * C;
    f->o_q1_b = o; o += f->H;
    f->o_q2_w = o; o += (long long)f->NO * f->H;
    f->o_q2_b = o; o += f->NO;
    f->npar = o;
    // host init: uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) for pointwise, scale/(C*C) * U[0,1) spectral
    std::vector<float> h((size_t)o, 0.f);
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    auto fill = [&](long long off, long long n, double lo, double hi) {
        for (long long i = 0; i < n; ++i) h[off + i] = (float)(lo + (hi - lo) * U(rng));
    };
    fill(f->o_lift_w, (long long)C * FI, -1.0 / std::sqrt(FI), 1.0 / std::sqrt(FI));
    for (int l = 0; l < L; ++l) {
        fill(f->o_R[l], 2LL * f->MODES * C * C, 0.0, 1.0 / ((double)C * C));
        fill(f->o_W[l], (long long)C * C, -1.0 / std::sqrt(C), 1.0 / std::sqrt(C));
    }
    fill(f->o_q1_w, (long long)f->H * C, -1.0 / std::sqrt(C), 1.0 / std::sqrt(C));
    fill(f->o_q2_w, (long long)f->NO * f->H, -1.0 / std::sqrt(f->H), 1.0 / std::sqrt(f->H));

    auto alloc = [&](float** p, long long n) -> bool {
        return cudaMalloc(p, (size_t)n * sizeof(float)) == cudaSuccess;
    };
    bool ok = alloc(&f->par, o) && alloc(&f->grad, o) && alloc(&f->m1, o) && alloc(&f->m2, o);
    // DFT matrices (float64 on the host, rounded once)
    const int NT = f->NT;
    std::vector<float> fx((size_t)P * 2 * m), by1((size_t)P * 2 * NT), by2((size_t)P * 2 * NT),
        bx1((size_t)m * P), bx2((size_t)m * P), bz1((size_t)NT * 2 * P), bz2((size_t)NT * 2 * P);
    for (int x = 0; x < P; ++x)
        for (int k = 0; k < m; ++k) {
            const double th = 2 * kPi * k * x / P;
            fx[(size_t)x * 2 * m + k] = (float)std::cos(th);
            fx[(size_t)x * 2 * m + m + k] = (float)(-std::sin(th));
        }
    // forward complex stage: out = re * [Cs | -Sn] + im * [Sn | Cs]  (kernel exp(-i th))
    for (int y = 0; y < P; ++y)
        for (int j = 0; j < NT; ++j) {
            const double th = 2 * kPi * freq_t(j, m, P) * y / P;
            by1[(size_t)y * 2 * NT + j] = (float)std::cos(th);
            by1[(size_t)y * 2 * NT + NT + j] = (float)(-std::sin(th));
            by2[(size_t)y * 2 * NT + j] = (float)std::sin(th);
            by2[(size_t)y * 2 * NT + NT + j] = (float)std::cos(th);
        }
    // inverse complex stage: out = re * [Cs | Sn] + im * [-Sn | Cs]  (kernel exp(+i th))
    for (int j = 0; j < NT; ++j)
        for (int z = 0; z < P; ++z) {
            const double th = 2 * kPi * freq_t(j, m, P) * z / P;
            bz1[(size_t)j * 2 * P + z] = (float)std::cos(th);
            bz1[(size_t)j * 2 * P + P + z] = (float)std::sin(th);
            bz2[(size_t)j * 2 * P + z] = (float)(-std::sin(th));
            bz2[(size_t)j * 2 * P + P + z] = (float)std::cos(th);
        }
    // inverse x: u = (1/P^3) sum_k w_k (re cos - im sin), w_0 = 1, w_k = 2
    const double inv = 1.0 / ((double)P * P * P);
    for (int k = 0; k < m; ++k)
        for (int x = 0; x < P; ++x) {
            const double th = 2 * kPi * k * x / P, w = (k == 0 ? 1.0 : 2.0) * inv;
            bx1[(size_t)k * P + x] = (float)(w * std::cos(th));
            bx2[(size_t)k * P + x] = (float)(-w * std::sin(th));
        }
    // the two matrices of a pair lie one behind the other: the adjoint stages take both
    // as one operand
    ok = ok && alloc(&f->Fx, fx.size()) && alloc(&f->By1, 2 * by1.size()) && alloc(&f->Bz1, 2 * bz1.size()) &&
         alloc(&f->Bx1, 2 * bx1.size());
    if (ok) {
        f->By2 = f->By1 + by1.size();
        f->Bz2 = f->Bz1 + bz1.size();
        f->Bx2 = f->Bx1 + bx1.size();
    }
    // activations for max batch
    const long long B = f->maxB, NV = f->NV;
    const long long nT1 = 2LL * m * B * C * P * P, nT2 = 2LL * NT * m * B * C * P, nT3 = 2LL * f->MODES * B * C;
    const long long nW1 = 2LL * P * NT * m * B * C, nW2 = 2LL * P * P * m * B * C;
    for (int l = 0; l <= L && ok; ++l) {
        float *a = nullptr, *z = nullptr;
        ok = alloc(&a, B * C * NV) && (l == 0 || alloc(&z, B * C * NV));   // (the lift has no pre-activation)
        f->act.push_back(a);
        f->pre.push_back(z);
    }
    for (int l = 0; l < L && ok; ++l) {
        float *t1, *t2, *t3, *u3, *w1, *w2;
        ok = alloc(&t1, nT1) && alloc(&t2, nT2) && alloc(&t3, nT3) && alloc(&u3, nT3) && alloc(&w1, nW1) && alloc(&w2, nW2);
        if (!ok) break;
        f->T1.push_back(t1); f->T2.push_back(t2); f->T3.push_back(t3); f->U3.push_back(u3);
        f->W1.push_back(w1); f->W2.push_back(w2);
    }
    long long big = std::max(std::max(nT1, nW2), B * C * NV);
    ok = ok && alloc(&f->feat, B * FI * NV) && alloc(&f->hq, B * f->H * NV) && alloc(&f->zq, B * f->H * NV) &&
         alloc(&f->out, B * f->NO * NV) && alloc(&f->gbuf0, std::max(B * f->H * NV, big)) &&
         alloc(&f->gbuf1, std::max(B * f->H * NV, big)) && alloc(&f->gT, std::max(big, nW1)) &&
         alloc(&f->gT2, std::max(big, nW1)) && alloc(&f->gout, B * f->NO * NV);
    ok = ok && cudaMalloc(&f->partial, 4096 * sizeof(double)) == cudaSuccess &&
         cudaMalloc(&f->bpart, (size_t)B * kRowChunks * std::max(std::max(C, f->H), f->NO) * sizeof(double)) == cudaSuccess;
    long long wmax = 0;
    for (auto mn : {std::pair<int, int>(f->NO, f->H), {f->H, C}, {C, C}, {C, FI}})
        wmax = std::max(wmax, (long long)wgrad_splits(mn.first, mn.second) * mn.first * mn.second);
    ok = ok && alloc(&f->wpart, wmax);
    if (!ok) {
        psatd_fno_destroy(f);
        return PSATD_ERR_OOM;
    }
    cudaStream_t s = f->stream;
    bool cp = cudaMemcpyAsync(f->par, h.data(), (size_t)o * sizeof(float), cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemsetAsync(f->m1, 0, (size_t)o * sizeof(float), s) == cudaSuccess &&
              cudaMemsetAsync(f->m2, 0, (size_t)o * sizeof(float), s) == cudaSuccess &&
              cudaMemcpyAsync(f->Fx, fx.data(), fx.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemcpyAsync(f->By1, by1.data(), by1.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemcpyAsync(f->By2, by2.data(), by2.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemcpyAsync(f->Bz1, bz1.data(), bz1.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemcpyAsync(f->Bz2, bz2.data(), bz2.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemcpyAsync(f->Bx1, bx1.data(), bx1.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemcpyAsync(f->Bx2, bx2.data(), bx2.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaStreamSynchronize(s) == cudaSuccess;
    if (!cp) {
        psatd_fno_destroy(f);
        return PSATD_ERR_CUDA;
    }
    *out = f;
    return PSATD_OK;
}

void psatd_fno_destroy(psatd_fno* f) {
    if (!f) return;
    if (f->stream) cudaStreamSynchronize(f->stream);
    float* ps[] = {f->par, f->grad, f->m1, f->m2, f->Fx, f->By1, f->Bz1, f->Bx1,
                   f->feat, f->hq, f->zq, f->out, f->gbuf0, f->gbuf1, f->gT, f->gT2, f->gout};
    for (float* p : ps)
        if (p) cudaFree(p);
    for (auto* v : {&f->act, &f->pre, &f->T1, &f->T2, &f->T3, &f->U3, &f->W1, &f->W2})
        for (float* p : *v)
            if (p) cudaFree(p);
    if (f->partial) cudaFree(f->partial);
    if (f->bpart) cudaFree(f->bpart);
    if (f->wpart) cudaFree(f->wpart);
    delete f;
}

long long psatd_fno_num_params(const psatd_fno* f) { return f ? f->npar : 0; }

psatd_status psatd_fno_buffers(psatd_fno* f, float** params, float** grads, float** output) {
    if (!f) return PSATD_ERR_ARG;
    if (params) *params = f->par;
    if (grads) *grads = f->grad;
    if (output) *output = f->out;
    return PSATD_OK;
}

const char* psatd_fno_last_error(const psatd_fno* f) { return f ? f->err.c_str() : "NULL model"; }

}  // extern "C"

namespace {

// Launches of the mixing kernels: shared memory for the staged spectra (sets, four
// bytes a value) and, backward through the input, as many weight rows as fit.
// A launch asks for up to LIMIT bytes.
template <int LIMIT, typename K>
cudaError_t mix_smem(K k, size_t bytes) {
    return bytes > 48 * 1024 ? allow_smem<LIMIT>(k) : cudaSuccess;
}
int mix_threads(int n) { return std::min(256, std::max(32, (n + 31) / 32 * 32)); }

cudaError_t mix_fwd(psatd_fno* f, const float* V, const float* R, float* U, int B) {
    if (B < 4) {
        mix_fwd_few_kernel<<<grid_for((long long)f->MODES * B * f->C), 256, 0, f->stream>>>(V, R, U, f->MODES, B, f->C);
        return cudaGetLastError();
    }
    const int items = (B + 3) / 4 * f->C;                          // of one mode
    const int per_block = std::max(1, 256 / items);
    const size_t need = (size_t)2 * per_block * B * f->C * sizeof(float);
    const int stage = need <= (size_t)kMixStage;
    const cudaError_t e = mix_smem<kMixStage>(mix_fwd_kernel, stage ? need : 0);
    if (e != cudaSuccess) return e;
    mix_fwd_kernel<<<(f->MODES + per_block - 1) / per_block, mix_threads(per_block * items), stage ? need : 0,
                     f->stream>>>(V, R, U, f->MODES, B, f->C, per_block, stage);
    return cudaGetLastError();
}

cudaError_t mix_back(psatd_fno* f, const float* gU, const float* V, const float* R, float* gR, float* gV, int B) {
    const int C = f->C;
    const size_t spec = (size_t)2 * B * C * sizeof(float);
    int stage = 2 * spec <= (size_t)kMixStage;
    cudaError_t e = mix_smem<kMixStage>(mix_back_weight_kernel, stage ? 2 * spec : 0);
    if (e != cudaSuccess) return e;
    mix_back_weight_kernel<<<f->MODES, mix_threads((C + 3) / 4 * C), stage ? 2 * spec : 0, f->stream>>>(
        gU, V, gR, f->MODES, B, C, stage);
    stage = spec <= (size_t)kMixStage;
    const size_t row = (size_t)2 * (C + 1) * sizeof(float);
    const int rows = (int)std::min<size_t>(C, kMixStage / row);
    const size_t bytes = (stage ? spec : 0) + rows * row;
    if ((e = mix_smem<2 * kMixStage>(mix_back_input_kernel, bytes)) != cudaSuccess) return e;
    mix_back_input_kernel<<<f->MODES, mix_threads((B + 3) / 4 * rows), bytes, f->stream>>>(gU, R, gV, f->MODES, B, C,
                                                                                         rows, stage);
    return cudaGetLastError();
}

// A product followed by a bias per row of C and, with gelu, the activation; the
// pre-activation is kept in C if `keep`.
GemmArgs with_bias(GemmArgs g, const float* bias, float* act, bool gelu, bool keep) {
    g.bias = bias;
    g.act = act;
    g.gelu = gelu;
    g.store_c = keep;
    return g;
}

// the complex stages: C = A B + A2 B2 (real and imaginary part)
GemmArgs paired(GemmArgs g, const float* A2, const float* B2) {
    g.A2 = A2;
    g.B2 = B2;
    return g;
}

// forward pass; with `train` it leaves the pre-activations for the backward pass
psatd_status fno_forward(psatd_fno* f, const float* prm, int B, bool train) {
    const int P = f->P, C = f->C, m = f->m, NT = f->NT, FI = f->NP + 3;
    const long long NV = f->NV;
    cudaStream_t s = f->stream;
    features_kernel<<<grid_for(B * FI * NV), 256, 0, s>>>(prm, f->NP, B, P, f->feat);
    // lift: act0[b] = W_lift (C x FI) feat[b] (FI x NV) + b_lift
    FCK(launch_gemm(with_bias(G(C, (int)NV, FI, f->par + f->o_lift_w, FI, 1, f->feat, NV, 1, f->act[0], NV, 1, 0.f, B, 0,
                                FI * NV, C * NV), f->par + f->o_lift_b, nullptr, false, true), s));
    for (int l = 0; l < f->L; ++l) {
        const float* v = f->act[l];
        float* z = f->pre[l + 1];
        const long long M1 = (long long)B * C * P * P;          // rows (b,c,z,y)
        // X: T1[(part,kx)][(b,c,z,y)] = v[(b,c,z,y)][x] Fx[x][(part,kx)]
        FCK(launch_gemm(G((int)M1, 2 * m, P, v, P, 1, f->Fx, 2 * m, 1, f->T1[l], 1, M1, 0.f), s));
        // Y: rows (kx,b,c,z) per part, contract y; out [(part,ky)][rows]
        const long long Mh = (long long)m * B * C * P;
        FCK(launch_gemm(paired(G((int)Mh, 2 * NT, P, f->T1[l], P, 1, f->By1, 2 * NT, 1, f->T2[l], 1, Mh, 0.f),
                               f->T1[l] + Mh * P, f->By2), s));
        // Z: rows (ky,kx,b,c) per part, contract z
        const long long Mz = (long long)NT * m * B * C;
        FCK(launch_gemm(paired(G((int)Mz, 2 * NT, P, f->T2[l], P, 1, f->By1, 2 * NT, 1, f->T3[l], 1, Mz, 0.f),
                               f->T2[l] + Mz * P, f->By2), s));
        // mode mixing: T3 = [part][kz][ky][kx][b][c] = [part][mode][b][c]
        FCK(mix_fwd(f, f->T3[l], f->par + f->o_R[l], f->U3[l], B));
        // Zi: rows r = (ky,kx,b,o), K = kz (stride Mz); out W1[(part,z)][r]
        FCK(launch_gemm(paired(G((int)Mz, 2 * P, NT, f->U3[l], 1, Mz, f->Bz1, 2 * P, 1, f->W1[l], 1, Mz, 0.f),
                               f->U3[l] + (long long)NT * Mz, f->Bz2), s));
        // Yi: W1[part][z][ky][Q], Q = (kx,b,o); batch z, rows Q, K = ky; out W2[(part,y)][z][Q]
        const long long Q = (long long)m * B * C;
        FCK(launch_gemm(paired(G((int)Q, 2 * P, NT, f->W1[l], 1, Q, f->Bz1, 2 * P, 1, f->W2[l], 1, (long long)P * Q, 0.f, P,
                                 (long long)NT * Q, 0, Q), f->W1[l] + (long long)P * NT * Q, f->Bz2), s));
        // Xi: W2[part][y][z][kx][(b,o)]; batch (y, z), rows (b,o), K = kx; out z[(b,o)][z][y][x]
        {
            GemmArgs g = G(B * C, P, m, f->W2[l], 1, (long long)B * C, f->Bx1, P, 1, z, NV, 1, 0.f);
            g.nb0 = P; g.nb1 = P;
            g.sAb0 = (long long)P * Q; g.sAb1 = Q;               // y, z
            g.sCb0 = P; g.sCb1 = (long long)P * P;
            FCK(launch_gemm(paired(g, f->W2[l] + (long long)P * P * Q, f->Bx2), s));
        }
        // pointwise W v added, bias and activation: z[b] += W (C x C) v[b] + b, act = GELU(z)
        // (the last layer has none, and its backward pass needs no z)
        const bool gelu = l + 1 < f->L;
        FCK(launch_gemm(with_bias(G(C, (int)NV, C, f->par + f->o_W[l], C, 1, v, NV, 1, z, NV, 1, 1.f, B, 0, C * NV,
                                    C * NV), f->par + f->o_b[l], f->act[l + 1], gelu, train && gelu), s));
    }
    // projection
    const int H = f->H, NO = f->NO;
    FCK(launch_gemm(with_bias(G(H, (int)NV, C, f->par + f->o_q1_w, C, 1, f->act[f->L], NV, 1, f->zq, NV, 1, 0.f, B, 0,
                                C * NV, H * NV), f->par + f->o_q1_b, f->hq, true, train), s));
    FCK(launch_gemm(with_bias(G(NO, (int)NV, H, f->par + f->o_q2_w, H, 1, f->hq, NV, 1, f->out, NV, 1, 0.f, B, 0,
                                H * NV, NO * NV), f->par + f->o_q2_b, nullptr, false, true), s));
    FCK(cudaGetLastError());
    return PSATD_OK;
}

// weight gradient gW (Mo x Ni) = sum_b gZ[b] (Mo x NV) * X[b]^T (NV x Ni)
cudaError_t weight_grad(psatd_fno* f, int Mo, int Ni, const float* gZ, const float* X, float* gW, int B) {
    const dim3 grid(wgrad_splits(Mo, Ni), (Mo + 31) / 32, (Ni + 31) / 32);
    wgrad_kernel<<<grid, 32 * kWgWarps, 0, f->stream>>>(gZ, X, B, Mo, Ni, f->NV, f->wpart);
    wgrad_reduce_kernel<<<(Mo * Ni + 7) / 8, 256, 0, f->stream>>>(f->wpart, (int)grid.x, Mo * Ni, gW);
    return cudaGetLastError();
}

// bias gradient of gz (no activation): gbias[c] = sum over b, v
cudaError_t bias_grad(psatd_fno* f, const float* gz, float* gbias, int B, int C) {
    act_back_kernel<false><<<B * C * kRowChunks, 256, 0, f->stream>>>(nullptr, gz, nullptr, B, C, f->NV, f->bpart);
    bias_reduce_kernel<<<C, 32, 0, f->stream>>>(f->bpart, B * kRowChunks, gbias);
    return cudaGetLastError();
}

// gz = ga * gelu'(z) and its bias gradient
cudaError_t gelu_back(psatd_fno* f, const float* z, const float* ga, float* gz, float* gbias, int B, int C) {
    act_back_kernel<true><<<B * C * kRowChunks, 256, 0, f->stream>>>(z, ga, gz, B, C, f->NV, f->bpart);
    bias_reduce_kernel<<<C, 32, 0, f->stream>>>(f->bpart, B * kRowChunks, gbias);
    return cudaGetLastError();
}

// An adjoint stage for both parts at once: columns n >= n of the second part lie
// part_stride elements after the first's.
GemmArgs both_parts(GemmArgs g, int n, long long part_stride) {
    g.nsplit = n;
    g.c_split = part_stride - n * g.sCn;
    return g;
}

psatd_status fno_backward(psatd_fno* f, int B) {
    const int P = f->P, C = f->C, m = f->m, NT = f->NT, H = f->H, NO = f->NO, FI = f->NP + 3;
    const long long NV = f->NV;
    cudaStream_t s = f->stream;
    float* g = f->grad;
    // output layer: gout holds dL/dout
    FCK(bias_grad(f, f->gout, g + f->o_q2_b, B, NO));
    FCK(weight_grad(f, NO, H, f->gout, f->hq, g + f->o_q2_w, B));
    // g_h = Wq2^T gout ; g_zq = g_h * gelu'(zq)
    FCK(launch_gemm(G(H, (int)NV, NO, f->par + f->o_q2_w, 1, H, f->gout, NV, 1, f->gbuf0, NV, 1, 0.f, B, 0, NO * NV,
                      H * NV), s));
    FCK(gelu_back(f, f->zq, f->gbuf0, f->gbuf0, g + f->o_q1_b, B, H));
    FCK(weight_grad(f, H, C, f->gbuf0, f->act[f->L], g + f->o_q1_w, B));
    // g_a(L) = Wq1^T g_zq
    float *ga = f->gbuf1, *other = f->gbuf0;
    FCK(launch_gemm(G(C, (int)NV, H, f->par + f->o_q1_w, 1, C, f->gbuf0, NV, 1, ga, NV, 1, 0.f, B, 0, H * NV, C * NV), s));
    for (int l = f->L - 1; l >= 0; --l) {
        // g_z = g_a * act'(z); the last layer has no activation: g_z is g_a, and the
        // gradient of its input goes to the other buffer
        float* gz = ga;
        if (l + 1 < f->L) {
            gz = other;
            FCK(gelu_back(f, f->pre[l + 1], ga, gz, g + f->o_b[l], B, C));
        } else {
            FCK(bias_grad(f, gz, g + f->o_b[l], B, C));
            std::swap(ga, other);
        }
        FCK(weight_grad(f, C, C, gz, f->act[l], g + f->o_W[l], B));
        // g_v (pointwise part) = W^T g_z -> ga (act[l] gradient), overwritten
        FCK(launch_gemm(G(C, (int)NV, C, f->par + f->o_W[l], 1, C, gz, NV, 1, ga, NV, 1, 0.f, B, 0, C * NV, C * NV), s));
        // spectral part, adjoint of Xi: g_W2[part] = gz (rows (b,o), per (y,z): x) * Bx^T
        const long long Q = (long long)m * B * C, Mz = (long long)NT * m * B * C, Mh = (long long)m * B * C * P;
        float* gW2 = f->gT;        // layout of W2
        {
            GemmArgs a = G(B * C, 2 * m, P, gz, NV, 1, f->Bx1, 1, P, gW2, 1, (long long)B * C, 0.f);
            a.nb0 = P; a.nb1 = P;
            a.sAb0 = P; a.sAb1 = (long long)P * P;              // gz[(b,o)][z][y][x]: y stride P, z stride P^2
            a.sCb0 = (long long)P * Q; a.sCb1 = Q;
            FCK(launch_gemm(both_parts(a, m, (long long)P * P * Q), s));
        }
        // adjoint of Yi: g_W1[part'] = sum over (part, y) of gW2 rows; W2 = W1re*Bz1 + W1im*Bz2
        float* gW1 = f->gT2;
        FCK(launch_gemm(both_parts(G((int)Q, 2 * NT, 2 * P, gW2, 1, (long long)P * Q, f->Bz1, 1, 2 * P, gW1, 1, Q, 0.f, P,
                                     Q, 0, (long long)NT * Q), NT, (long long)P * NT * Q), s));
        // adjoint of Zi: g_U[part'] rows (ky,kx,b,o), K over (part,z) of gW1
        float* gU = f->gT;
        FCK(launch_gemm(both_parts(G((int)Mz, 2 * NT, 2 * P, gW1, 1, Mz, f->Bz1, 1, 2 * P, gU, 1, Mz, 0.f), NT,
                                   (long long)NT * Mz), s));
        // mixing: weights and spectra
        float* gV = f->gT2;
        FCK(mix_back(f, gU, f->T3[l], f->par + f->o_R[l], g + f->o_R[l], gV, B));
        // adjoint of Z: g_T2[part] (rows (ky,kx,b,c), K = z) = gV (rows, 2NT) * By_part^T
        float* gT2 = f->gT;
        FCK(launch_gemm(both_parts(G((int)Mz, 2 * P, 2 * NT, gV, 1, Mz, f->By1, 1, 2 * NT, gT2, P, 1, 0.f), P, Mz * P), s));
        // adjoint of Y: g_T1[part] (rows (kx,b,c,z), K = y)
        float* gT1 = f->gT2;
        FCK(launch_gemm(both_parts(G((int)Mh, 2 * P, 2 * NT, gT2, 1, Mh, f->By1, 1, 2 * NT, gT1, P, 1, 0.f), P, Mh * P), s));
        // adjoint of X: g_v += gT1 (rows (b,c,z,y), 2m) * Fx^T
        const long long M1 = (long long)B * C * P * P;
        FCK(launch_gemm(G((int)M1, P, 2 * m, gT1, 1, M1, f->Fx, 1, 2 * m, ga, P, 1, 1.f), s));
    }
    // lift
    FCK(bias_grad(f, ga, g + f->o_lift_b, B, C));
    FCK(weight_grad(f, C, FI, ga, f->feat, g + f->o_lift_w, B));
    FCK(cudaGetLastError());
    return PSATD_OK;
}

}  // namespace

extern "C" {

psatd_status psatd_fno_forward(psatd_fno* f, const float* params_dev, int batch, float* out_dev) {
    if (!f || !params_dev || batch < 1 || batch > f->maxB) return fno_fail(f, PSATD_ERR_ARG, "bad arguments");
    psatd_status st = fno_forward(f, params_dev, batch, false);
    if (st) return st;
    if (out_dev && out_dev != f->out) {
        FCK(cudaMemcpyAsync(out_dev, f->out, (size_t)batch * f->NO * f->NV * sizeof(float), cudaMemcpyDeviceToDevice,
                            f->stream));
    }
    return PSATD_OK;
}

psatd_status psatd_fno_loss_backward(psatd_fno* f, const float* params_dev, int batch, const float* target_dev,
                                     double* loss) {
    if (!f || !params_dev || !target_dev || batch < 1 || batch > f->maxB)
        return fno_fail(f, PSATD_ERR_ARG, "bad arguments");
    psatd_status st = fno_forward(f, params_dev, batch, true);
    if (st) return st;
    const long long n = (long long)batch * f->NO * f->NV;
    const int nb = std::min(4096, grid_for(n));
    mse_kernel<<<nb, 256, 0, f->stream>>>(f->out, target_dev, f->gout, n, f->partial);
    st = fno_backward(f, batch);
    if (st) return st;
    if (loss) {
        std::vector<double> h(nb);
        FCK(cudaMemcpyAsync(h.data(), f->partial, nb * sizeof(double), cudaMemcpyDeviceToHost, f->stream));
        FCK(cudaStreamSynchronize(f->stream));
        double s = 0;
        for (double v : h) s += v;
        *loss = s / (double)n;
    }
    return PSATD_OK;
}

psatd_status psatd_fno_adam_step(psatd_fno* f, float lr, float beta1, float beta2, float eps, float weight_decay) {
    if (!f) return PSATD_ERR_ARG;
    f->adam_t += 1;
    const float c1 = 1.f - std::pow(beta1, (float)f->adam_t), c2 = 1.f - std::pow(beta2, (float)f->adam_t);
    adam_kernel<<<grid_for(f->npar), 256, 0, f->stream>>>(f->par, f->grad, f->m1, f->m2, f->npar, lr, beta1, beta2, eps,
                                                           weight_decay, c1, c2);
    FCK(cudaGetLastError());
    return PSATD_OK;
}

psatd_status psatd_gemm_bf16(int M, int N, int K, const float* A, long long sAm, long long sAk, const float* B,
                             long long sBk, long long sBn, float* C, long long sCm, long long sCn, float alpha,
                             float beta, int ksplit, void* cuda_stream) {
    if (!A || !B || !C || M < 0 || N < 0 || K < 0) return PSATD_ERR_ARG;
    GemmArgs g = G(M, N, K, A, sAm, sAk, B, sBk, sBn, C, sCm, sCn, beta);
    g.alpha = alpha;
    g.ksplit = ksplit < 1 ? 1 : ksplit;
    return launch_gemm(g, static_cast<cudaStream_t>(cuda_stream)) == cudaSuccess ? PSATD_OK : PSATD_ERR_CUDA;
}

psatd_status psatd_gemm_bf16_tma(int M, int N, int K, const void* A, const void* B, float* C, void* cuda_stream) {
    if (!A || !B || !C) return PSATD_ERR_ARG;
    const cudaError_t e = launch_gemm_tma(A, B, C, M, N, K, static_cast<cudaStream_t>(cuda_stream));
    if (e == cudaErrorInvalidValue) return PSATD_ERR_ARG;
    return e == cudaSuccess ? PSATD_OK : PSATD_ERR_CUDA;
}

psatd_status psatd_gemm_synchronize(void* cuda_stream) {
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return PSATD_ERR_CUDA;
    return gemm_take_error() ? PSATD_ERR_TIMEOUT : PSATD_OK;
}

psatd_status psatd_fno_synchronize(psatd_fno* f) {
    if (!f) return PSATD_ERR_ARG;
    FCK(cudaStreamSynchronize(f->stream));
    if (gemm_take_error()) return fno_fail(f, PSATD_ERR_TIMEOUT, "a bounded wait in the tensor-core GEMM expired");
    return PSATD_OK;
}

}  // extern "C"
