// Persistent batched PSATD advance: many periodic boxes (pulse realisations on
// grids of different sizes) stepped together in ONE cooperative launch.
//
// A step of every box is the same five phases (Sec. 2.1, Eq. 3-4 between the
// forward and inverse 3D DFTs): x forward, y forward, the fused z pass (z
// forward, the per-mode update, z inverse), y inverse, x inverse.  Each phase is
// one list of work items over all boxes (box p owns items [pre[p], pre[p+1])),
// which the resident blocks draw one at a time from a global ticket counter
// (a block that drew small items takes more); a grid-wide barrier separates the
// phases, because a phase reads what every block wrote in the one before.  The
// launch runs n steps, i.e. 5 n - 1 barriers, without returning to the host;
// a box with fewer steps of its own skips its items in the later steps.
//
// Work items:
//   x: W_x consecutive rows of one box (contiguous in memory);
//   y: W_y consecutive x-columns at one (component, z);
//   z: W_z consecutive x-columns at one y, all six components: forward z
//      transforms, the update of every mode of the tile, inverse z transforms.
// Any axis length with factors 2, 3, 5 runs the in-place passes of fft_mixed.cuh with
// radices up to 16; the radix schedule of each axis and the three tile widths come
// from the host (the batch autotuner picks them per axis length).  In float32 a length
// of two such radices, at the untuned tile widths, runs the compile-time tiles of
// fft_two.cuh instead (MultiProblem::two), which leave out the run-time index
// arithmetic: 16 sweep boxes of 96 to 192 points an axis, two to three steps, 11.2 ms
// with the run-time passes, 9.45 ms with these (five sweeps of the boxes at the
// copy bandwidth take 5.6 ms).
//
// The barrier: every block adds one to a global counter after a fence, and
// thread 0 polls the counter (acquire loads, a short sleep between polls) until
// it reaches the number of arrivals that barrier needs.  The wait is bounded by
// the global nanosecond timer; a block whose wait expires sets
// DEV_ERR_GRID_TIMEOUT in the device error word and leaves the kernel, and so
// does every other block at the next barrier it cannot pass, so no block spins
// forever.  Field loads go around L1 (cache-global) so that no block reads a
// line another block rewrote in the previous phase.
#include "fft_mixed.cuh"
#include "fft_two.cuh"
#include "tma.cuh"

namespace psatd {

namespace {

constexpr int kMT = 256;

template <typename T> constexpr size_t desc_bytes() { return (sizeof(MultiProblem<T>) + 127) / 128 * 128; }

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier number `target / gridDim.x` (see above); false if this block's
// wait expired.
__device__ bool grid_barrier(unsigned* bar, unsigned target, int* err, unsigned long long limit_ns) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        const unsigned long long t0 = global_ns();
        int done = 0;
        for (unsigned it = 0; it < (1u << 30); ++it) {
            if (ld_acquire_gpu(bar) >= target) {
                done = 1;
                break;
            }
            if (global_ns() - t0 > limit_ns) break;
            __nanosleep(128);
        }
        if (!done) atomicOr(err, DEV_ERR_GRID_TIMEOUT);
        __threadfence();
        ok = done;
    }
    __syncthreads();
    return ok != 0;
}

// x phase: rows row0 .. row0 + nrow - 1 of the box ([6][Nz][Ny] rows of Nx).
template <typename T, int S>
__device__ __forceinline__ void x_tile(const MultiProblem<T>& P, long long item, cplx<T>* sm) {
    const int Nx = P.N[0], W = P.W[0];
    const long long rows = 6LL * P.N[1] * P.N[2], row0 = item * W;
    MixTile<T> t;
    t.base = P.f + row0 * Nx;
    t.buf = GBuf<cplx<T>>{P.f, rows * Nx};
    t.cstride = 0;
    t.stride = 1;
    t.logw = 0;
    t.nw = (int)min((long long)W, rows - row0);
    t.nq = 1;
    t.slot = 0;
    t.P = row_stride(Nx, P.plan[0].radix[0]);
    t.run = row_run(Nx, P.plan[0].radix[0]);
    t.gap = t.run - Nx / P.plan[0].radix[0];
    mix_transform<T, S, kNarrow, true, true>(t, sm, P.plan[0], P.tp[0]);
}

// y phase: x-columns x0 .. x0 + nw - 1 of plane (comp, z).
template <typename T, int S>
__device__ __forceinline__ void y_tile(const MultiProblem<T>& P, long long item, cplx<T>* sm) {
    const int Nx = P.N[0], Ny = P.N[1], Nz = P.N[2], W = P.W[1];
    const int ntile = (Nx + W - 1) / W;
    const unsigned rest = (unsigned)item / (unsigned)ntile;                   // comp * Nz + z
    const int tile = (int)((unsigned)item - rest * ntile);
    const long long plane = (long long)Nx * Ny;
    const int x0 = tile * W;
    MixTile<T> t;
    t.base = P.f + rest * plane + x0;
    t.buf = GBuf<cplx<T>>{P.f, 6LL * plane * Nz};
    t.cstride = 0;
    t.stride = Nx;
    t.logw = 31 - __clz(W);
    t.nw = min(W, Nx - x0);
    t.nq = 1;
    t.slot = 0;
    t.P = t.run = t.gap = 0;
    mix_transform<T, S, kNarrow, false, true>(t, sm, P.plan[1], P.tp[1]);
}

// z phase: x-columns x0 .. x0 + nw - 1 at one y, all six components: forward z
// transforms, the update of every mode on the digit-reversed spectra, inverse z
// transforms.
template <typename T>
__device__ __forceinline__ void z_tile(const MultiProblem<T>& P, long long item, cplx<T>* sm) {
    const int Nx = P.N[0], Ny = P.N[1], Nz = P.N[2], W = P.W[2], logw = 31 - __clz(W);
    const int ntile = (Nx + W - 1) / W;
    const int y = (int)((unsigned)item / (unsigned)ntile), tile = (int)item - y * ntile, x0 = tile * W, ct = Nz << logw;
    const long long plane = (long long)Nx * Ny, cstride = plane * Nz;
    MixTile<T> t;
    t.base = P.f + (long long)y * Nx + x0;
    t.buf = GBuf<cplx<T>>{P.f, 6LL * cstride};
    t.cstride = cstride;
    t.stride = plane;
    t.logw = logw;
    t.nw = min(W, Nx - x0);
    t.nq = 6;
    t.slot = ct;
    t.P = t.run = t.gap = 0;
    mix_forward<T, kNarrow, true>(t, sm, P.plan[2], P.tp[2]);

    const int Nxh = Nx / 2 + 1, Nyh = Ny / 2 + 1;
    const int ay = min(y, Ny - y);
    const T ky = P.k[1][PSATD_IX(y, Ny)];
    const long long ncoef = (long long)(Nz / 2 + 1) * Nyh * Nxh;
    for (int e = threadIdx.x; e < ct; e += blockDim.x) {
        const int c = e & (W - 1), n = mix_frequency(P.plan[2], e >> logw);
        if (c >= t.nw) continue;
        const int ix = x0 + c;
        const int ax = min(ix, Nx - ix), az = min(n, Nz - n);
        const ModeCoef<T> m = P.coef[PSATD_IX(((size_t)az * Nyh + ay) * Nxh + ax, ncoef)];
        cplx<T>* o = sm + e;
        cplx<T> Ex = o[0], Ey = o[ct], Ez = o[2 * ct], Bx = o[3 * ct], By = o[4 * ct], Bz = o[5 * ct];
        rotate_mode<T>(Ex, Ey, Ez, Bx, By, Bz, P.k[0][PSATD_IX(ix, Nx)] * m.kinv, ky * m.kinv,
                       P.k[2][PSATD_IX(n, Nz)] * m.kinv, m.C, m.S);
        o[0] = Ex; o[ct] = Ey; o[2 * ct] = Ez;
        o[3 * ct] = Bx; o[4 * ct] = By; o[5 * ct] = Bz;
    }
    __syncthreads();
    mix_inverse<T, kNarrow>(t, sm, P.plan[2], P.tp[2]);
}

// ---------------------------------------------------------------------------
// float32 lengths of two radices up to 16: the compile-time tiles of fft_two.cuh,
// each a function of its own, with the tile at its fixed place in shared memory.  As
// calls they keep the kernel at 80 registers (three blocks an SM; 16 bytes of spills in
// the kernel's own frame) and cost a jump an item, which is 2 us of work or more.
__device__ __forceinline__ float2* multi_tile() {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    return reinterpret_cast<float2*>(smem_raw + desc_bytes<float>());
}

template <int R1, int R2, int S>
__device__ __noinline__ void x_two(const MultiProblem<float>& P, int item) {
    constexpr int G = TwoCfg<R1, R2>::G;
    const long long rows = 6LL * P.N[1] * P.N[2], row0 = (long long)item * G;
    two_rows_tile<R1, R2, S, true>(P.f + row0 * (R1 * R2), (int)min((long long)G, rows - row0), P.tp[0], multi_tile(),
                                   GBuf<float2>{P.f, rows * (R1 * R2)});
}

template <int R1, int R2, int S>
__device__ __noinline__ void y_two(const MultiProblem<float>& P, int item) {
    const int Nx = P.N[0], ntile = (Nx + kTwoW - 1) / kTwoW;
    const unsigned rest = (unsigned)item / (unsigned)ntile;                    // comp * Nz + z
    const int x0 = ((int)((unsigned)item - rest * ntile)) * kTwoW, c = threadIdx.x % kTwoW, t = threadIdx.x / kTwoW;
    const long long plane = (long long)Nx * (R1 * R2);
    two_cols_tile<R1, R2, S, true>(P.f + rest * plane + x0 + c, (size_t)Nx, t, c, x0 + c < Nx, P.tp[1], multi_tile(),
                                   GBuf<float2>{P.f, 6LL * plane * P.N[2]});
}

template <int R1, int R2>
__device__ __noinline__ void z_two(const MultiProblem<float>& P, int item) {
    constexpr int W = kTwoKW, N = R1 * R2, SLOT = N * W;
    float2* sm = multi_tile();
    const int Nx = P.N[0], Ny = P.N[1], ntile = (Nx + W - 1) / W;
    const int y = (int)((unsigned)item / (unsigned)ntile), x0 = (item - y * ntile) * W, nw = min(W, Nx - x0);
    const size_t plane = (size_t)Nx * Ny, cstride = plane * N;
    float2* base = P.f + (size_t)y * Nx + x0;
    const GBuf<float2> F{P.f, 6LL * (long long)cstride};
    two_z_forward<R1, R2, kMT, true>(base, plane, cstride, nw, P.tp[2], sm, F);
    const int Nxh = Nx / 2 + 1, Nyh = Ny / 2 + 1, ay = min(y, Ny - y);
    const float ky = P.k[1][PSATD_IX(y, Ny)];
    const long long ncoef = (long long)(N / 2 + 1) * Nyh * Nxh;
#pragma unroll 1
    for (int e = threadIdx.x; e < SLOT; e += kMT) {
        const int c = e % W, pos = e / W, k1 = pos / R2, n = k1 + (pos - k1 * R2) * R1;
        if (c >= nw) continue;
        const int ix = x0 + c, ax = min(ix, Nx - ix), az = min(n, N - n);
        const ModeCoef<float> m = P.coef[PSATD_IX(((size_t)az * Nyh + ay) * Nxh + ax, ncoef)];
        float2* o = sm + e;
        float2 Ex = o[0], Ey = o[SLOT], Ez = o[2 * SLOT], Bx = o[3 * SLOT], By = o[4 * SLOT], Bz = o[5 * SLOT];
        rotate_mode<float>(Ex, Ey, Ez, Bx, By, Bz, P.k[0][PSATD_IX(ix, Nx)] * m.kinv, ky * m.kinv,
                           P.k[2][PSATD_IX(n, N)] * m.kinv, m.C, m.S);
        o[0] = Ex; o[SLOT] = Ey; o[2 * SLOT] = Ez;
        o[3 * SLOT] = Bx; o[4 * SLOT] = By; o[5 * SLOT] = Bz;
    }
    __syncthreads();
    two_z_inverse<R1, R2, kMT>(base, plane, cstride, nw, P.tp[2], sm, F);
}

// (longer z tiles are over the budget and take the run-time passes)
template <int R1, int R2>
__device__ __forceinline__ void two_phase_z(const MultiProblem<float>& P, int item) {
    if constexpr (6 * R1 * R2 * kTwoKW * sizeof(float2) <= multi_tile_budget<float>()) z_two<R1, R2>(P, item);
}

// Phase ph of the item with the compile-time tile `id`.
__device__ __forceinline__ void two_phase(int ph, int id, const MultiProblem<float>& P, int item) {
    switch (id) {
#define PSATD_TWO_CASE(i, r1, r2)                            \
    case i:                                                  \
        if (ph == 0) x_two<r1, r2, -1>(P, item);             \
        else if (ph == 1) y_two<r1, r2, -1>(P, item);        \
        else if (ph == 2) two_phase_z<r1, r2>(P, item);      \
        else if (ph == 3) y_two<r1, r2, +1>(P, item);        \
        else x_two<r1, r2, +1>(P, item);                     \
        break;
        PSATD_TWO_PAIRS(PSATD_TWO_CASE)
#undef PSATD_TWO_CASE
        default: break;
    }
}

// float32: three blocks per SM (room for 85 registers a thread, tiles of at most 72 KB)
template <typename T>
__global__ void __launch_bounds__(kMT, sizeof(T) == 4 ? 3 : 2)
multi_advance_kernel(const MultiProblem<T>* __restrict__ probs, const long long* __restrict__ prefix, int nprob,
                     int nsteps, unsigned* bar, unsigned long long* ticket, int* err, unsigned long long limit_ns,
                     unsigned extra) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    MultiProblem<T>* P = reinterpret_cast<MultiProblem<T>*>(smem_raw);
    cplx<T>* tile = reinterpret_cast<cplx<T>*>(smem_raw + desc_bytes<T>());
    __shared__ long long s_item;
    int cur = -1;                                               // box whose descriptor is in P
    unsigned nbar = 0;
    unsigned long long base = 0;                                // first ticket of this phase
    for (int s = 0; s < nsteps; ++s) {
        for (int ph = 0; ph < 5; ++ph) {
            const int a = ph <= 2 ? ph : 4 - ph;               // axis of the phase: x, y, z, y, x
            const long long* pre = prefix + (size_t)a * (nprob + 1);
            const long long total = pre[nprob];
            // items are handed out one at a time from a global ticket counter, so
            // blocks that drew cheap items (small boxes) take more of them; every
            // block stops at its first ticket past the phase, so the phase uses
            // exactly total + gridDim.x tickets.  Thread 0 draws the next ticket when
            // an item begins, so the counter's round trip (about 1 us against 2 to 3 us
            // for a tile) is over when the item ends.
            unsigned long long drawn = 0;
            if (threadIdx.x == 0) s_item = (long long)(atomicAdd(ticket, 1ull) - base);
            __syncthreads();
            for (;;) {
                const long long g = s_item;
                if (g >= total) break;
                if (threadIdx.x == 0) drawn = atomicAdd(ticket, 1ull);
                int lo = 0, hi = nprob - 1;                     // the box p with pre[p] <= g < pre[p + 1]
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (pre[PSATD_IX(mid, nprob + 1)] <= g) lo = mid;
                    else hi = mid - 1;
                }
                if (lo != cur) {
                    const int* src = reinterpret_cast<const int*>(probs + lo);
                    int* dst = reinterpret_cast<int*>(P);
                    for (int i = threadIdx.x; i < (int)(sizeof(MultiProblem<T>) / 4); i += blockDim.x) dst[i] = src[i];
                    cur = lo;
                    __syncthreads();
                }
                const long long item = g - pre[lo];
                bool done = s >= P->nsteps;                     // a box past its own step count is skipped
                if constexpr (sizeof(T) == 4) {
                    if (!done && P->two[a] >= 0) {
                        two_phase(ph, P->two[a], *P, (int)item);
                        done = true;
                    }
                }
                if (!done) {
                    if (ph == 0) x_tile<T, -1>(*P, item, tile);
                    else if (ph == 1) y_tile<T, -1>(*P, item, tile);
                    else if (ph == 2) z_tile<T>(*P, item, tile);
                    else if (ph == 3) y_tile<T, +1>(*P, item, tile);
                    else x_tile<T, +1>(*P, item, tile);
                }
                __syncthreads();                                // every thread has read s_item, the descriptor and the tile
                if (threadIdx.x == 0) s_item = (long long)(drawn - base);
                __syncthreads();
            }
            __syncthreads();                                    // s_item is read before the next phase writes it
            base += (unsigned long long)total + gridDim.x;
            if (s == nsteps - 1 && ph == 4) return;
            ++nbar;
            if (!grid_barrier(bar, nbar * gridDim.x + extra, err, limit_ns)) return;
        }
    }
}

}  // namespace

template <typename T>
size_t multi_tile_bytes(int axis, const AxisPlan& pl, int W) {
    const size_t es = sizeof(cplx<T>);
    return (size_t)W * es * (axis == 0 ? (size_t)row_stride(pl.N, pl.radix[0]) : (size_t)(axis == 2 ? 6 : 1) * pl.N);
}

template <typename T>
cudaError_t launch_multi_advance(const MultiProblem<T>* probs, const long long* prefix, int nprob, int nsteps,
                                 size_t tile_bytes, long long max_items, unsigned* bar, int* err,
                                 unsigned long long limit_ns, unsigned extra, cudaStream_t s, int* grid_out) {
    auto k = multi_advance_kernel<T>;
    const size_t smem = desc_bytes<T>() + tile_bytes;
    cudaError_t e = allow_smem<(int)(desc_bytes<T>() + multi_tile_budget<T>())>(k);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kMT, smem)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    long long grid = (long long)per_sm * sms;
    if (max_items < grid) grid = max_items < 1 ? 1 : max_items;
    // barrier counter at bar[0], ticket counter at bar[2] (8-byte aligned)
    unsigned long long* ticket = reinterpret_cast<unsigned long long*>(bar + 2);
    if ((e = cudaMemsetAsync(bar, 0, 16, s)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(kMT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;            // all blocks resident at once (the barrier needs it)
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (grid_out) *grid_out = (int)grid;
    return cudaLaunchKernelEx(&cfg, k, probs, prefix, nprob, nsteps, bar, ticket, err, limit_ns, extra);
}

template size_t multi_tile_bytes<float>(int, const AxisPlan&, int);
template size_t multi_tile_bytes<double>(int, const AxisPlan&, int);
template cudaError_t launch_multi_advance<float>(const MultiProblem<float>*, const long long*, int, int, size_t,
                                                 long long, unsigned*, int*, unsigned long long, unsigned,
                                                 cudaStream_t, int*);
template cudaError_t launch_multi_advance<double>(const MultiProblem<double>*, const long long*, int, int, size_t,
                                                  long long, unsigned*, int*, unsigned long long, unsigned,
                                                  cudaStream_t, int*);

}  // namespace psatd
