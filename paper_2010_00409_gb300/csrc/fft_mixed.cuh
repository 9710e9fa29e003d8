// Mixed-radix transforms of pencils staged in shared memory, for every axis
// length with factors 2, 3 and 5 (the forward DFT is exp(-2 pi i nk/N), S = -1;
// the inverse S = +1; neither is normalised).
//
// N is split into as few radices as possible, each a register DFT of up to 16
// (or 32) points: one or two passes for nearly every length to 1024 instead of
// the three or four of radices 2, 3, 4, 5 and 8.  The first pass reads its
// operands straight from global memory and the last writes its results there,
// so a two-pass transform touches shared memory twice per value (one store, one
// load) where staged passes of small radices touch it eight times.
//
// The passes are in place (decimation in frequency).  Level p has blocks of M
// points (M = N at first), radix R and L = M / R: item (block, j < L) takes the R
// values at block * M + j + r L, forms their R-point DFT and multiplies output k
// by W_M^{jk}, and stores it at block * M + k L + j, the positions it read.  So no
// pass needs a second buffer or a barrier between its loads and its stores.
// After the last level position k1 L1 + k2 L2 + ... + kn holds the frequency
// k1 + R1 k2 + R1 R2 k3 + ...; the last pass stores to that index, and the fused
// k-space pass works on the digit-reversed spectrum and runs the levels backwards
// (decimation in time) for the inverse.
//
// Twiddles come from a table in position order, W_M^{jk} at k L + j of its level
// (levels one after another, below 2 N entries), so neighbouring items read
// neighbouring entries.
//
// Layouts in shared memory: columns (y, z): position * W + column, W a power of
// two, the lanes of a warp on consecutive columns; rows (x): row * P + position,
// the first level's R runs of L values spaced an odd number of values apart
// (row_run), so the last pass, whose lanes read one run each, spreads over the banks.
// All the values of an item are a constant step apart in either memory, so an
// access costs one or two address additions (with the padding and 64-bit products
// worked out per access the y pass of a 180 x 135 x 150 box issued 91 instructions
// per value, about half of them addresses).
#pragma once

#include "fft_reg.cuh"

namespace psatd {

constexpr int kNarrow = 16, kWide = 32;        // largest radix of the two kernel variants

// Division by a plan's constant d as a multiply-high: q = umulhi(n, m) with
// m = ceil(2^32 / d) equals n / d for 0 <= n < 2^16 and 1 <= d < 2^16 (the
// error term n (m - 2^32/d) / 2^32 < 2^-16 stays below the gap 1/d to the next
// integer); d = 1 has m = 0 and is taken apart.
__host__ __device__ __forceinline__ unsigned div_multiplier(int d) {
    return d <= 1 ? 0u : 0xFFFFFFFFu / (unsigned)d + 1u;
}

// Rows: the spacing of the first level's runs, and a row's values in all.
__host__ __device__ __forceinline__ int row_run(int N, int R0) { return (N / R0) | 1; }
__host__ __device__ __forceinline__ int row_stride(int N, int R0) { return R0 * row_run(N, R0) | 1; }
// Padded rows (PAD below): float32 plans of three levels, radices to 16, the last a multiple of 8.
// The last pass's lanes read that many consecutive values each, so an even spacing puts
// half a warp on one or two banks (2048 = 16 x 16 x 8: eight ways); a spare value behind
// each such block spreads them, and runs R values apart mod 16 line the middle pass's
// blocks of R lanes up behind each other.  2048 x 64 x 64 step 1208 -> 1092 us, 1536 x
// 64 x 64 812 -> 776 us.  In float64, bound by its pipe, it changes nothing.
__host__ __device__ __forceinline__ bool row_padded(const AxisPlan& pl) {
    return pl.npass == 3 && pl.radix[0] <= kNarrow && pl.radix[2] % 8 == 0;
}
__host__ __device__ __forceinline__ int row_run_padded(const AxisPlan& pl) {
    const int R = pl.radix[2], n = pl.N / pl.radix[0], run = n + n / R;
    return run + ((R - run) & 15);
}

// Position-ordered twiddle entries of a plan (all levels but the last, whose
// twiddles are 1).
__host__ __device__ inline int mix_table_size(const AxisPlan& pl) {
    int n = 0, M = pl.N;
    for (int p = 0; p + 1 < pl.npass; ++p) {
        n += M;
        M /= pl.radix[p];
    }
    return n;
}

#ifdef __CUDACC__
__device__ __forceinline__ int fdiv(int n, unsigned m) { return m == 0u ? n : (int)__umulhi((unsigned)n, m); }

// The frequency of last-level block u: the digits k1 .. k(n-1) of u reversed.
__device__ __forceinline__ int mix_natural(const AxisPlan& pl, int u) {
    if (pl.npass <= 2) return u;                    // one digit or none
    int k = 0, L = pl.N / pl.radix[pl.npass - 1], w = 1;
    for (int p = 0; p + 1 < pl.npass; ++p) {
        L /= pl.radix[p];
        const int d = u / L;
        u -= d * L;
        k += d * w;
        w *= pl.radix[p];
    }
    return k;
}
// The frequency held at position pos after the last level.
__device__ __forceinline__ int mix_frequency(const AxisPlan& pl, int pos) {
    if (pl.npass <= 2) {                            // one run per first digit: pos = k1 R2 + k2, k = k1 + R1 k2
        const int u = fdiv(pos, pl.div_run), run = pl.N / pl.radix[0];
        return pl.npass < 2 ? pos : u + (pos - u * run) * pl.radix[0];
    }
    const int R = pl.radix[pl.npass - 1], u = pos / R;
    return mix_natural(pl, u) + (pos - u * R) * (pl.N / R);
}

// Where a block's pencils lie.  Columns: value n of column c of component q at
// base[q cstride + n stride + c] (c < nw <= W = 2^logw), and at q slot + n W + c in
// shared memory.  Rows: value n of row w at base[w N + n] (w < nw), and in shared
// memory at w P, run by run (run values apart).
template <typename T> struct MixTile {
    cplx<T>* base;
    GBuf<cplx<T>> buf;
    long long cstride, stride;
    int logw, nw, nq, slot, P, run, gap;             // gap = run - N / radix[0]
};

// One level over the tile's pencils.  DIF: from_g loads the operands from global
// memory (first level), to_g stores the results to their frequency there (last
// level).  DIT (the levels backwards): operands from shared memory, to_g stores to
// global memory (first level).  CG: global loads go around L1 (values other SMs
// wrote during this launch).
// PAD (rows): the padded layout of row_run_padded.
template <typename T, int S, int R, bool ROWS, bool DIT, bool CG, bool PAD>
__device__ __forceinline__ void mix_pass(const MixTile<T>& t, cplx<T>* sm, const AxisPlan& pl, int p, int M,
                                         const cplx<T>* __restrict__ tp, bool from_g, bool to_g) {
    const int N = pl.N, nb = N / R, L = M / R;                  // (divisions by a compile-time R)
    const unsigned dnb = pl.div_nb[p], dl = pl.div_l[p];
    const int items = ROWS ? t.nw * nb : (t.nq * nb) << t.logw;
    for (int b = threadIdx.x; b < items; b += blockDim.x) {
        int u, c, q = 0;
        if constexpr (ROWS) {
            c = fdiv(b, dnb);
            u = b - c * nb;
        } else {
            c = b & ((1 << t.logw) - 1);
            u = b >> t.logw;
            if (t.nq > 1) {
                q = fdiv(u, dnb);
                u -= q * nb;
            }
            if (c >= t.nw) continue;
        }
        const int blk = fdiv(u, dl), j = u - blk * L;
        const int pos0 = blk * M + j;
        // the item's R values in shared memory: s0 + r ss
        cplx<T>* s0;
        int ss;
        if constexpr (ROWS) {
            // first level: value r in run r; deeper levels lie inside one run
            if (p == 0) {
                s0 = sm + c * t.P + j;
                if constexpr (PAD) s0 += fdiv(j, pl.div_l[1]);          // (the last radix is the second level's L)
                ss = t.run;
            } else {
                const int run0 = fdiv(pos0, pl.div_run);
                s0 = sm + c * t.P + pos0 + run0 * t.gap;
                if constexpr (PAD) s0 += p == 1 ? blk * R : blk;        // last-level blocks before pos0
                ss = PAD && p == 1 ? L + 1 : L;
            }
        } else {
            s0 = sm + q * t.slot + (pos0 << t.logw) + c;
            ss = L << t.logw;
        }
        cplx<T>* grow = ROWS ? t.base + (long long)c * N : t.base + q * t.cstride + c;
        cplx<T> v[R];
        if (!DIT && from_g) {
            const cplx<T>* gp = ROWS ? grow + pos0 : grow + pos0 * t.stride;
            const long long gs = ROWS ? (long long)L : L * t.stride;
            static_for<0, R>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                if constexpr (CG) v[r] = __ldcg(&t.buf.at(gp, 0));
                else v[r] = t.buf.at(gp, 0);
                gp += gs;
            });
        } else {
            const cplx<T>* sp = s0;
            static_for<0, R>([&](auto rc) {
                v[decltype(rc)::value] = *sp;
                sp += ss;
            });
        }
        if (DIT && L > 1) {
            int at = L + j;
            static_for<1, R>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                const cplx<T> w = tp[PSATD_IX(at, M)];
                v[r] = S < 0 ? cmul(v[r], w) : cmulc(v[r], w);
                at += L;
            });
        }
        reg_dft<T, S, R>(v);
        if (!DIT && L > 1) {
            int at = L + j;
            static_for<1, R>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                const cplx<T> w = tp[PSATD_IX(at, M)];
                v[r] = S < 0 ? cmul(v[r], w) : cmulc(v[r], w);
                at += L;
            });
        }
        if (to_g) {
            const int n0 = DIT ? pos0 : mix_natural(pl, blk), dn = DIT ? L : nb;
            cplx<T>* gp = ROWS ? grow + n0 : grow + n0 * t.stride;
            const long long gs = ROWS ? (long long)dn : dn * t.stride;
            static_for<0, R>([&](auto rc) {
                t.buf.at(gp, 0) = v[decltype(rc)::value];
                gp += gs;
            });
        } else {
            cplx<T>* sp = s0;
            static_for<0, R>([&](auto rc) {
                *sp = v[decltype(rc)::value];
                sp += ss;
            });
        }
    }
}

template <typename T, int S, int MAXR, bool ROWS, bool DIT, bool CG, bool PAD = false>
__device__ __forceinline__ void mix_dispatch(const MixTile<T>& t, cplx<T>* sm, const AxisPlan& pl, int p, int M,
                                             const cplx<T>* tp, bool from_g, bool to_g) {
    const int R = pl.radix[p];
#define PSATD_MIX(r) \
    case r: mix_pass<T, S, r, ROWS, DIT, CG, PAD>(t, sm, pl, p, M, tp, from_g, to_g); return
    switch (R) {
        PSATD_MIX(1); PSATD_MIX(2); PSATD_MIX(3); PSATD_MIX(4); PSATD_MIX(5); PSATD_MIX(6); PSATD_MIX(8);
        PSATD_MIX(9); PSATD_MIX(10); PSATD_MIX(12); PSATD_MIX(15); PSATD_MIX(16);
        default: break;
    }
    if constexpr (MAXR > kNarrow) {
        switch (R) {
            PSATD_MIX(18); PSATD_MIX(20);
            default: break;
        }
    }
    if constexpr (MAXR > kNarrow && sizeof(T) == 4) {             // (float64 plans stop at 20)
        switch (R) {
            PSATD_MIX(24); PSATD_MIX(25); PSATD_MIX(27); PSATD_MIX(30); PSATD_MIX(32);
            default: break;
        }
    }
#undef PSATD_MIX
}

// The whole transform of a tile from global to global memory.  Called by the whole
// block; ends without a barrier (the last pass reads shared memory).
template <typename T, int S, int MAXR, bool ROWS, bool CG, bool PAD = false>
__device__ __forceinline__ void mix_transform(const MixTile<T>& t, cplx<T>* sm, const AxisPlan& pl,
                                              const cplx<T>* tp) {
    int M = pl.N;
#pragma unroll 1
    for (int p = 0; p < pl.npass; ++p) {
        if (p > 0) __syncthreads();
        mix_dispatch<T, S, MAXR, ROWS, false, CG, PAD>(t, sm, pl, p, M, tp, p == 0, p == pl.npass - 1);
        tp += M;
        M /= pl.radix[p];
    }
}

// Forward transform of a tile (columns) from global memory into shared memory, the
// spectrum in digit-reversed order; ends with a barrier.
template <typename T, int MAXR, bool CG>
__device__ __forceinline__ void mix_forward(const MixTile<T>& t, cplx<T>* sm, const AxisPlan& pl, const cplx<T>* tp) {
    int M = pl.N;
#pragma unroll 1
    for (int p = 0; p < pl.npass; ++p) {
        mix_dispatch<T, -1, MAXR, false, false, CG>(t, sm, pl, p, M, tp, p == 0, false);
        __syncthreads();
        tp += M;
        M /= pl.radix[p];
    }
}

// Inverse transform of the digit-reversed spectra in shared memory to global
// memory; ends without a barrier.
template <typename T, int MAXR>
__device__ __forceinline__ void mix_inverse(const MixTile<T>& t, cplx<T>* sm, const AxisPlan& pl, const cplx<T>* tp) {
    int M = 1, off = mix_table_size(pl);
#pragma unroll 1
    for (int p = pl.npass - 1; p >= 0; --p) {
        M *= pl.radix[p];
        if (p < pl.npass - 1) {
            off -= M;
            __syncthreads();
        }
        mix_dispatch<T, +1, MAXR, false, true, false>(t, sm, pl, p, M, tp + off, false, p == 0);
    }
}
#endif

}  // namespace psatd
