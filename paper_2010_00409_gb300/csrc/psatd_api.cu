// C ABI of the PSATD library (declared in include/psatd.h): argument checks,
// axis tables, device memory, and the order of kernel launches.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include <cudaTypedefs.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>

#include "../../include/psatd.h"
#include "common.cuh"
#include "fft_mixed.cuh"
#include "fft_two.cuh"
#include "tma.cuh"

using namespace psatd;

namespace psatd {

#ifdef PSATD_DEBUG
void debug_register_reader(long long (*reader)(long long*, long long*));
#endif

namespace {
const int kRadices[] = {32, 30, 27, 25, 24, 20, 18, 16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};

// Extend cur (radices so far, non-increasing) by a factorisation of n; best keeps
// the fewest passes, then the smallest largest radix, then the smallest sum.
void search_plan(int n, int max_radix, AxisPlan* cur, int sum, AxisPlan* best, int* best_sum) {
    if (n == 1) {
        const bool first = best->npass == 0;
        if (first || cur->npass < best->npass ||
            (cur->npass == best->npass && (cur->radix[0] < best->radix[0] ||
                                           (cur->radix[0] == best->radix[0] && sum < *best_sum)))) {
            *best = *cur;
            *best_sum = sum;
        }
        return;
    }
    if (cur->npass >= (best->npass ? best->npass : kMaxPass)) return;
    for (int r : kRadices) {
        if (r > max_radix || n % r) continue;
        cur->radix[cur->npass++] = r;
        search_plan(n / r, r, cur, sum + r, best, best_sum);
        --cur->npass;
    }
}

std::vector<AxisPlan> plan_table(int max_radix) {
    std::vector<AxisPlan> t(2049);
    for (int N = 0; N <= 2048; ++N) {
        AxisPlan cur{}, best{};
        int n = N, sum = 0;
        for (int f : {2, 3, 5})
            while (n > 1 && n % f == 0) n /= f;
        cur.N = best.N = N;
        if (N == 1) {
            best.npass = 1;
            best.radix[0] = 1;
        } else if (N > 1 && n == 1) {
            search_plan(N, max_radix, &cur, 0, &best, &sum);
        }
        finish_plan(&best);
        t[N] = best;
    }
    return t;
}
}  // namespace

void finish_plan(AxisPlan* p) {
    int M = p->N;
    for (int i = 0; i < p->npass; ++i) {
        p->div_nb[i] = div_multiplier(p->N / p->radix[i]);
        p->div_l[i] = div_multiplier(M / p->radix[i]);
        M /= p->radix[i];
    }
    p->div_run = p->npass ? div_multiplier(p->N / p->radix[0]) : 0u;
}

bool make_plan(int N, AxisPlan* p, int max_radix) {
    static const std::vector<AxisPlan> t16 = plan_table(16), t20 = plan_table(20), t32 = plan_table(32);
    if (N < 1 || N > 2048) return false;
    *p = (max_radix >= 32 ? t32 : max_radix >= 20 ? t20 : t16)[N];
    return p->npass > 0;
}

// The plan of a context's axis (0 x, 1 y, 2 z): radices beyond 16 only where they save
// a pass.  In float64 a wide kernel takes all the registers of an SM for one block, so
// along x and y three narrow passes beat two wide ones (step of 64 x 360 x 64 2.67 ->
// 2.39 ms, 360 x 64 x 64 2.61 -> 2.39 ms, 2000 x 64 x 64 16.4 -> 15.3 ms); along z, where
// a pass fewer is a trip of six components through shared memory and back, radices to
// 20 stay where they make two passes (64 x 64 x 162: 6 % faster so).
// In float32 two radices up to 16 are never joined into one of 18 to 32 points: one
// pass has an item a pencil, half a warp in a 16-column block, and the two
// compile-time passes of fft_two.cuh are faster for all seven such lengths in the mean
// (a step of 32^3 points 50.4 -> 12.7 us, 24^3 30.4 -> 11.2 us, 240 x 250 x 25 220 ->
// 155 us, 20 x 240 x 250 185 -> 138 us; the other way 1000 x 27 x 90 334 -> 341 us).
bool context_plan(int N, int precision, int axis, AxisPlan* p) {
    AxisPlan wide;
    if (!make_plan(N, p) || !make_plan(N, &wide, precision == 64 ? 20 : 32)) return false;
    const bool take = precision == 64 ? axis == 2 && wide.npass == 2 : p->npass > 2;
    if (take && wide.npass < p->npass) *p = wide;
    return true;
}

}  // namespace psatd

namespace {

constexpr double kTwoPi = 6.28318530717958647692;
constexpr int kMaxN = 2048;
constexpr int kDiagBlocks = 1024;

thread_local std::string g_create_error = "no error";

// autotuner results per (Nx, Ny, Nz, precision): kernel path and tile shift
std::map<std::tuple<int, int, int, int>, std::pair<int, int>> g_tuned;
std::mutex g_tuned_mutex;

struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
};

}  // namespace

struct psatd_batch {
    cudaStream_t stream = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    bool capturing = false;
    cudaError_t capture_error = cudaSuccess;
    std::vector<std::pair<psatd_ctx*, double>> time_advance;   // per replay: ctx time += value
    std::vector<std::pair<psatd_ctx*, double>> time_set;       // per replay: ctx time = value
};

namespace {
thread_local psatd_batch* g_capture = nullptr;   // batch being captured on this thread
}

struct psatd_ctx {
    psatd_grid grid{};
    psatd_mapping mapping{};
    double dt = 0.0;
    double t = 0.0;
    int prec = 32;
    cudaStream_t stream = nullptr;
    int device = 0;

    // fields
    void* fields = nullptr;
    size_t field_bytes = 0;
    bool own_fields = false;
    bool real_fields = false;           // real float32 storage (PSATD_FLAG_REAL_FIELDS)
    DevBuf slot_k, slot_coef;           // real fields: k_x per slot, coefficient table in slot order
    DevBuf slot_mode;                   // real fields: x mode index per slot (sampling from the half spectrum)
    DevBuf slot_coef_proj;              // real fields: projection table (C = 1/Ntot, S = 0) in slot order
    DevBuf nyq;                         // real fields: x Nyquist spectrum [6][Nz][Ny] between the plane kernels
    DevBuf tw2[3];                      // N_a = 512 / 1024: [32][32] twiddles of the register kernels
    CUtensorMap nyq_map;                // ... and its tensor map for the k-space kernel (128-B aligned type)
    bool nyq_map_ok = false;

    // tables (device)
    DevBuf tw[3], k[3], coef;
    // position-ordered twiddles of the context's plan, then of the batched advance's
    // radix schedules (values from each one's start)
    DevBuf twp[3];
    int twp_at[3][3] = {{0}};
    AxisPlan plan[3];

    // longitudinal profile of PSATD_PULSE_PROFILE pulses (psatd_set_pulse_profile)
    DevBuf lprof;
    int lprof_n = 0;
    double lprof_z0 = 0.0, lprof_dz = 0.0;

    // scratch (device), allocated on first use
    DevBuf diag_spec, diag_partial, diag_out;
    DevBuf diag_nyq;                    // real fields: the x-Nyquist array of the diagnostics' spectrum
    DevBuf samp_wx, samp_wy, samp_wz, samp_g, samp_h, samp_out;
    int samp_ny = 0, samp_nz = 0;

    long long launches = 0;
    int kernel_path = PSATD_PATH_AUTO;
    int tile_shift = 0;                 // generic-kernel tile width scale (autotuner)

    // tensor map of the field storage for the copy-engine-fed k-space kernel
    CUtensorMap field_map;              // (the type is 128-byte aligned)
    void* field_map_ptr = nullptr;      // storage the map was encoded for
    bool field_map_real = false;        // ... and whether as a real-field half spectrum
    bool field_map_ok = false;
    int* dev_err = nullptr;             // device error word (bits of psatd::DeviceError)

    // one-shot focal path: coefficient table for one step of T, and a flag set
    // while the field storage holds an updated spectrum instead of the field
    DevBuf coef_T;
    double coef_T_step = 0.0;
    bool coef_T_ok = false;
    DevBuf coef_proj;                   // C = 1/Ntot, S = 0: the projection through the TMA kernel
    bool holds_spectrum = false;

    // persistent batched advance led by this context: barrier counter, work
    // prefix and box descriptors on the device, and the bytes last uploaded
    DevBuf multi;
    std::vector<unsigned char> multi_sig;
    std::string err = "no error";

    // per-kernel event timing (psatd_profile_enable)
    struct Pending { cudaEvent_t a, b; int kind; };
    bool prof_on = false;
    std::vector<cudaEvent_t> ev_pool;
    std::vector<Pending> pending;
    double prof_ms[PSATD_KERNEL_KINDS] = {0};
    long long prof_n[PSATD_KERNEL_KINDS] = {0};
};

namespace {

psatd_status fail(psatd_ctx* c, psatd_status s, const std::string& msg) {
    if (c) c->err = msg;
    else g_create_error = msg;
    return s;
}

psatd_status cuda_fail(psatd_ctx* c, cudaError_t e, const char* where) {
    std::string m = std::string(where) + ": " + cudaGetErrorString(e);
    return fail(c, e == cudaErrorMemoryAllocation ? PSATD_ERR_OOM : PSATD_ERR_CUDA, m);
}

// ---------------------------------------------------------------------------
// Failure injection for host-side tests (psatd_debug_*): a cap on the bytes of
// device memory the library holds (an allocation past it fails as cudaMalloc
// would, without calling it), and an armed CUDA error that replaces the result
// of the n-th checked call from now (the call itself is skipped).
std::mutex g_alloc_mutex;
std::map<void*, size_t> g_alloc_sizes;
long long g_alloc_live = 0;
long long g_alloc_limit = -1;                     // -1: no cap
std::atomic<int> g_inject_after{0};               // 0: nothing armed
std::atomic<int> g_inject_error{0};

#ifdef PSATD_DEBUG
std::mutex g_dbg_mutex;
std::vector<long long (*)(long long*, long long*)>& dbg_readers() {
    static std::vector<long long (*)(long long*, long long*)> r;
    return r;
}
#endif
}  // namespace

#ifdef PSATD_DEBUG
void psatd::debug_register_reader(long long (*reader)(long long*, long long*)) {
    std::lock_guard<std::mutex> lock(g_dbg_mutex);
    dbg_readers().push_back(reader);
}
#endif

namespace {

cudaError_t lib_malloc(void** p, size_t bytes) {
    std::lock_guard<std::mutex> lock(g_alloc_mutex);
    if (g_alloc_limit >= 0 && g_alloc_live + (long long)bytes > g_alloc_limit) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaSuccess) {
        g_alloc_sizes[*p] = bytes;
        g_alloc_live += (long long)bytes;
    }
    return e;
}

void lib_free(void* p) {
    if (!p) return;
    cudaFree(p);
    std::lock_guard<std::mutex> lock(g_alloc_mutex);
    auto it = g_alloc_sizes.find(p);
    if (it != g_alloc_sizes.end()) {
        g_alloc_live -= (long long)it->second;
        g_alloc_sizes.erase(it);
    }
}

// True (once) when the armed error is due at this checked call.
bool inject_due() {
    int n = g_inject_after.load();
    while (n > 0) {
        if (g_inject_after.compare_exchange_weak(n, n - 1)) return n == 1;
    }
    return false;
}

#define CK(ctx, call)                                                                        \
    do {                                                                                     \
        cudaError_t e_ = inject_due() ? (cudaError_t)g_inject_error.load() : (call);         \
        if (e_ != cudaSuccess) return cuda_fail((ctx), e_, #call);                           \
    } while (0)

size_t cplx_size(int prec) { return prec == 64 ? 16 : 8; }
size_t n_cells(const psatd_grid& g) { return (size_t)g.Nx * g.Ny * g.Nz; }
// bytes of one stored field value
size_t value_size(const psatd_ctx* c) { return c->real_fields ? sizeof(float) : cplx_size(c->prec); }

void free_buf(DevBuf& b) {
    if (b.p) lib_free(b.p);
    b.p = nullptr;
    b.bytes = 0;
}

cudaError_t ensure_buf(DevBuf& b, size_t bytes) {
    if (b.p && b.bytes >= bytes) return cudaSuccess;
    free_buf(b);
    cudaError_t e = lib_malloc(&b.p, bytes);
    if (e == cudaSuccess) b.bytes = bytes;
    else b.p = nullptr;
    return e;
}

bool is_finite(double v) { return std::isfinite(v); }

GridGeom geom(const psatd_ctx* c) {
    GridGeom g;
    g.Nx = c->grid.Nx; g.Ny = c->grid.Ny; g.Nz = c->grid.Nz;
    g.dx = c->grid.dx; g.dy = c->grid.dy; g.dz = c->grid.dz;
    g.x_min = c->grid.x_min; g.y_min = c->grid.y_min; g.z_min = c->grid.z_min;
    g.c = c->grid.c;
    return g;
}

template <typename T>
Tables<T> tables(const psatd_ctx* c) {
    Tables<T> tb;
    tb.tile_shift = c->tile_shift;
    for (int a = 0; a < 3; ++a) {
        tb.tw[a] = static_cast<const cplx<T>*>(c->tw[a].p);
        tb.k[a] = static_cast<const T*>(c->k[a].p);
        tb.plan[a] = c->plan[a];
        tb.twp[a] = static_cast<const cplx<T>*>(c->twp[a].p) + c->twp_at[a][0];
        tb.twn[a] = static_cast<const cplx<T>*>(c->twp[a].p) + c->twp_at[a][1];
    }
    tb.coef = static_cast<const ModeCoef<T>*>(c->coef.p);
    for (int a = 0; a < 3; ++a) tb.tw2[a] = static_cast<const cplx<T>*>(c->tw2[a].p);
    return tb;
}

// Radix schedules the batch autotuner chooses from for an axis of N points: the
// radices of make_plan (up to 16) largest first (0) or smallest first (1).
constexpr int kPlanVariants = 2;
bool make_plan_variant(int N, int variant, AxisPlan* p) {
    if (!make_plan(N, p)) return false;
    if (variant & 1) {
        std::reverse(p->radix, p->radix + p->npass);
        finish_plan(p);
    }
    return true;
}

int axis_n(const psatd_grid& g, int a) { return a == 0 ? g.Nx : (a == 1 ? g.Ny : g.Nz); }
double axis_d(const psatd_grid& g, int a) { return a == 0 ? g.dx : (a == 1 ? g.dy : g.dz); }

// signed index m of position i in numpy fftfreq order
int freq_index(int i, int N) { return i <= (N - 1) / 2 ? i : i - N; }

template <typename T>
psatd_status upload_axis_tables(psatd_ctx* c) {
    for (int a = 0; a < 3; ++a) {
        const int N = axis_n(c->grid, a);
        const double d = axis_d(c->grid, a);
        std::vector<cplx<T>> tw(N);
        std::vector<T> k(N);
        for (int t = 0; t < N; ++t) {
            const double ang = kTwoPi * (double)t / (double)N;
            if constexpr (sizeof(T) == 4) {
                const UnitF w = unit_f32(std::cos(ang), -std::sin(ang));
                tw[t] = mk<T>(w.c, w.s);
            } else {
                tw[t] = mk<T>((T)std::cos(ang), (T)(-std::sin(ang)));
            }
            k[t] = (T)(kTwoPi * (double)freq_index(t, N) / (N * d));
        }
        CK(c, ensure_buf(c->tw[a], N * sizeof(cplx<T>)));
        CK(c, ensure_buf(c->k[a], N * sizeof(T)));
        CK(c, cudaMemcpy(c->tw[a].p, tw.data(), N * sizeof(cplx<T>), cudaMemcpyHostToDevice));
        CK(c, cudaMemcpy(c->k[a].p, k.data(), N * sizeof(T), cudaMemcpyHostToDevice));
        // position-ordered twiddles: level p (blocks of M, radix R, L = M / R) holds
        // W_M^{jk} at k L + j
        std::vector<cplx<T>> tp;
        for (int v = -1; v < kPlanVariants; ++v) {
            AxisPlan pl = c->plan[a];
            if (v >= 0) make_plan_variant(N, v, &pl);
            c->twp_at[a][v + 1] = (int)tp.size();
            int M = N;
            for (int p = 0; p + 1 < pl.npass; ++p) {
                const int R = pl.radix[p], L = M / R;
                for (int kk = 0; kk < R; ++kk)
                    for (int j = 0; j < L; ++j) tp.push_back(tw[(size_t)j * kk % M * (N / M)]);
                M = L;
            }
        }
        if (tp.empty()) tp.push_back(tw[0]);
        CK(c, ensure_buf(c->twp[a], tp.size() * sizeof(cplx<T>)));
        CK(c, cudaMemcpy(c->twp[a].p, tp.data(), tp.size() * sizeof(cplx<T>), cudaMemcpyHostToDevice));
        if (N == 512 || N == 1024) {
            // the register kernels read W^{i j} for i, j < 32 along a thread-indexed j
            std::vector<cplx<T>> t2(32 * 32);
            for (int i = 0; i < 32; ++i)
                for (int j = 0; j < 32; ++j) t2[i * 32 + j] = tw[(i * j) % N];
            CK(c, ensure_buf(c->tw2[a], t2.size() * sizeof(cplx<T>)));
            CK(c, cudaMemcpy(c->tw2[a].p, t2.data(), t2.size() * sizeof(cplx<T>), cudaMemcpyHostToDevice));
        } else {
            free_buf(c->tw2[a]);
        }
    }
    return PSATD_OK;
}

// The table (C/Ntot, S/Ntot, 1/|k|) per |m| octant of one step dt into dst (or
// the step's table), in stream order.  slot_order: column p < Nx/2 holds the x
// mode of half-spectrum slot p (real fields), column Nx/2 the x Nyquist mode.
// projection: C = 1/Ntot, S = 0 (with the B projection of the k-space kernel this
// is the one-time transverse projection).  wait: return when the table is in
// memory; the tensor-copy-fed k-space kernel reads it before its wait on the
// previous kernel, so a table whose build no ordinary launch separates from that
// kernel is waited for here.
// A stream that is being captured is refused: the table belongs to the context,
// and a replay would rewrite it under calls that rely on another step.
template <typename T>
psatd_status upload_coef(psatd_ctx* c, double dt, DevBuf* dst = nullptr, bool slot_order = false,
                         bool projection = false, bool wait = true) {
    DevBuf& buf = dst ? *dst : c->coef;
    const psatd_grid& g = c->grid;
    const size_t n = (size_t)(g.Nx / 2 + 1) * (g.Ny / 2 + 1) * (g.Nz / 2 + 1);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CK(c, cudaStreamIsCapturing(c->stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) return cuda_fail(c, cudaErrorStreamCaptureUnsupported, "coefficient table");
    CK(c, ensure_buf(buf, n * sizeof(ModeCoef<T>)));
    CK(c, launch_coef<T>(static_cast<ModeCoef<T>*>(buf.p), geom(c), dt, projection,
                         slot_order ? static_cast<const int*>(c->slot_mode.p) : nullptr, c->stream));
    if (wait) CK(c, cudaStreamSynchronize(c->stream));
    return PSATD_OK;
}

psatd_status set_coef(psatd_ctx* c, double dt) {
    psatd_status st = c->prec == 64 ? upload_coef<double>(c, dt) : upload_coef<float>(c, dt);
    if (st == PSATD_OK && c->real_fields) st = upload_coef<float>(c, dt, &c->slot_coef, true);
    return st;
}

psatd_batch* capturing(const psatd_ctx* c);

psatd_status check_ctx(psatd_ctx* c, bool need_fields, bool need_physical = false) {
    if (!c) return fail(nullptr, PSATD_ERR_ARG, "NULL context");
    if (need_fields && !c->fields) return fail(c, PSATD_ERR_STATE, "no field storage bound");
    if (need_physical && c->holds_spectrum)
        return fail(c, PSATD_ERR_STATE, "storage holds the one-shot spectrum; set the field or a pulse first");
    cudaError_t e = cudaSetDevice(c->device);
    if (e != cudaSuccess) return cuda_fail(c, e, "cudaSetDevice");
    return PSATD_OK;
}

cudaEvent_t take_event(psatd_ctx* c) {
    if (!c->ev_pool.empty()) {
        cudaEvent_t e = c->ev_pool.back();
        c->ev_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    return e;
}

// Move finished (or, with wait, the oldest `upto`) event pairs into the totals.
cudaError_t harvest(psatd_ctx* c, size_t upto) {
    size_t i = 0;
    for (; i < c->pending.size() && i < upto; ++i) {
        auto& p = c->pending[i];
        cudaError_t e = cudaEventSynchronize(p.b);
        if (e != cudaSuccess) return e;
        float ms = 0.f;
        e = cudaEventElapsedTime(&ms, p.a, p.b);
        if (e != cudaSuccess) return e;
        c->prof_ms[p.kind] += ms;
        c->prof_n[p.kind] += 1;
        c->ev_pool.push_back(p.a);
        c->ev_pool.push_back(p.b);
    }
    c->pending.erase(c->pending.begin(), c->pending.begin() + i);
    return cudaSuccess;
}

// Run one launch (or a group of launches) of kernel kind `kind` inside an NVTX
// range named for the kind (visible to Nsight tools; a no-op without one), and
// bracketed by events when profiling is on.
struct NvtxRange {
    explicit NvtxRange(int kind) { nvtxRangePushA(psatd_kernel_name(kind)); }
    ~NvtxRange() { nvtxRangePop(); }
};

template <typename F>
cudaError_t timed(psatd_ctx* c, int kind, F&& launch) {
    NvtxRange range(kind);
    if (!c->prof_on) return launch();
    cudaEvent_t a = take_event(c), b = take_event(c);
    if (!a || !b) return cudaErrorMemoryAllocation;
    cudaError_t e = cudaEventRecord(a, c->stream);
    if (e != cudaSuccess) return e;
    e = launch();
    if (e != cudaSuccess) return e;
    e = cudaEventRecord(b, c->stream);
    if (e != cudaSuccess) return e;
    c->pending.push_back({a, b, kind});
    if (c->pending.size() > 8192) return harvest(c, 4096);
    return cudaSuccess;
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        cudaGetLastError();
        return PFN_cuTensorMapEncodeTiled_v12000(nullptr);
    }();
    return fn;
}

// (Re)encode the field tensor map when the storage changed; false if the
// copy-engine path does not apply to this grid.
bool ensure_field_map(psatd_ctx* c) {
    if (c->field_map_ptr == c->fields && c->field_map_real == c->real_fields) return c->field_map_ok;
    c->field_map_ptr = c->fields;
    c->field_map_real = c->real_fields;
    c->field_map_ok = false;
    const psatd_grid& g = c->grid;
    if (g.Nz > 256 || !c->dev_err) return false;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t es = cplx_size(c->prec), xw = es / 8;
    const cuuint64_t nx = c->real_fields ? g.Nx / 2 : g.Nx;     // complex values per stored row
    const cuuint64_t dims[4] = {nx * xw, (cuuint64_t)g.Ny, (cuuint64_t)g.Nz, 6};
    const cuuint64_t strides[3] = {nx * es, nx * g.Ny * es, nx * g.Ny * g.Nz * es};
    const int bz = kspace_tma_box_z(g.Nz);
    if (bz == 0) return false;
    const cuuint32_t box[4] = {(cuuint32_t)kspace_tma_box_x(c->prec), 1, (cuuint32_t)bz, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    if (dims[0] < box[0] || (nx * es) % 16 != 0) return false;
    CUresult r = enc(&c->field_map, CU_TENSOR_MAP_DATA_TYPE_INT64, 4, c->fields, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    c->field_map_ok = (r == CUDA_SUCCESS);
    return c->field_map_ok;
}

// The batch capturing this context's stream, if any.
psatd_batch* capturing(const psatd_ctx* c) {
    return (g_capture && g_capture->capturing && g_capture->stream == c->stream) ? g_capture : nullptr;
}

// Read and clear the device error word (synchronises the stream).
psatd_status check_device_error(psatd_ctx* c) {
    if (!c->dev_err) return PSATD_OK;
    int h = 0;
    CK(c, cudaMemcpyAsync(&h, c->dev_err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    CK(c, cudaStreamSynchronize(c->stream));
    if (h) {
        CK(c, cudaMemsetAsync(c->dev_err, 0, sizeof(int), c->stream));
        CK(c, cudaStreamSynchronize(c->stream));
        if (h & DEV_ERR_GRID_TIMEOUT)
            return fail(c, PSATD_ERR_TIMEOUT, "a bounded grid-barrier wait of the persistent batched advance expired; "
                                              "the fields of its boxes are invalid");
        return fail(c, PSATD_ERR_TIMEOUT, "a bounded device wait for a tensor copy expired; results of that step are invalid");
    }
    return PSATD_OK;
}

}  // namespace

const TwoPassEntry* psatd::two_pass_entry(int N) {
    const TwoPassEntry* (*const parts[])(int) = {two_pass_part0, two_pass_part1, two_pass_part2, two_pass_part3,
                                                 two_pass_part4, two_pass_part5, two_pass_part6, two_pass_part7};
    for (auto part : parts)
        if (const TwoPassEntry* e = part(N)) return e;
    return nullptr;
}

namespace {

// The compile-time two-pass transform of one axis; cudaErrorNotSupported (nothing
// launched) for float64 and lengths without one.
template <typename T>
cudaError_t fft_axis_two(cplx<T>* data, int ncomp, const GridGeom& g, const Tables<T>& tb, int axis, int dir,
                         cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        const AxisPlan& pl = tb.plan[axis];
        const TwoPassEntry* e = two_pass_entry(pl.N);
        if (!e || pl.npass != 2 || pl.radix[0] != e->R1) return cudaErrorNotSupported;
        const TwoPassArgs a{data, tb.twp[axis], axis, g.Nx, g.Ny, g.Nz, ncomp};
        const long long blocks =
            axis == 0 ? ((long long)ncomp * g.Nz * g.Ny + e->rows_per_block - 1) / e->rows_per_block
                      : (long long)ncomp * (axis == 1 ? g.Nz : g.Ny) * ((g.Nx + 15) / 16);
        if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
        auto k = axis == 0 ? e->rows[dir > 0] : e->cols[dir > 0];
        if (!k) return cudaErrorNotSupported;
        const int smem = axis == 0 ? e->rows_smem : e->cols_smem;
        if (smem > 48 * 1024) {
            const cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (r != cudaSuccess) return r;
        }
        return launch_pdl(k, dim3((unsigned)blocks), dim3(axis == 0 ? e->rows_threads : e->cols_threads), (size_t)smem, s,
                          a);
    }
    return cudaErrorNotSupported;
}

// The compile-time fused k-space pass (any KspaceMode), as above.
template <typename T>
cudaError_t kspace_two(cplx<T>* data, const GridGeom& g, const Tables<T>& tb, int mode, double scale, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        const AxisPlan& pl = tb.plan[2];
        const TwoPassEntry* e = two_pass_entry(pl.N);
        if (!e || !e->kspace || pl.npass != 2 || pl.radix[0] != e->R1) return cudaErrorNotSupported;
        const TwoPassArgs a{data, tb.twp[2], 2, g.Nx, g.Ny, g.Nz, 6};
        const TwoPassModes m{tb.k[0], tb.k[1], tb.k[2], tb.coef, mode, (float)scale};
        const cudaError_t r = cudaFuncSetAttribute(e->kspace, cudaFuncAttributeMaxDynamicSharedMemorySize, e->kspace_smem);
        if (r != cudaSuccess) return r;
        return launch_pdl(e->kspace, dim3((unsigned)((long long)g.Ny * ((g.Nx + 7) / 8))), dim3(e->kspace_threads),
                          (size_t)e->kspace_smem, s, a, m);
    }
    return cudaErrorNotSupported;
}

template <typename T>
cudaError_t fft_axis(psatd_ctx* c, cplx<T>* data, int ncomp, int axis, int dir, int kind) {
    const GridGeom g = geom(c);
    const Tables<T> tb = tables<T>(c);
    if (c->plan[axis].N <= 1) return cudaSuccess;
    return timed(c, kind < 0 ? axis : kind, [&] {
        if (c->kernel_path != PSATD_PATH_GENERIC) {
            cudaError_t e = launch_fft_axis_fast<T>(data, ncomp, g, tb, axis, dir, c->stream);
            if (e == cudaErrorNotSupported) e = fft_axis_two<T>(data, ncomp, g, tb, axis, dir, c->stream);
            if (e != cudaErrorNotSupported) {
                ++c->launches;
                return e;
            }
        }
        return launch_fft_axis<T>(data, ncomp, g, tb, axis, dir, c->stream, &c->launches);
    });
}

// Fused x+y plane transform when the cluster kernel covers this plane shape
// (AUTO path); returns cudaErrorNotSupported otherwise.
template <typename T>
cudaError_t plane_xy(psatd_ctx* c, cplx<T>* data, int ncomp, int dir, int kind) {
    const GridGeom g = geom(c);
    if (c->kernel_path != PSATD_PATH_AUTO || !plane_xy_supported(c->prec, g)) return cudaErrorNotSupported;
    const Tables<T> tb = tables<T>(c);
    return timed(c, kind < 0 ? (int)PSATD_KERNEL_PLANE_XY : kind, [&] {
        ++c->launches;
        return launch_plane_xy<T>(data, ncomp, g, tb, dir, c->stream);
    });
}

template <typename T>
cudaError_t fft3d(psatd_ctx* c, cplx<T>* data, int ncomp, int dir, int kind = -1) {
    cudaError_t e;
    if (dir < 0) {
        e = plane_xy<T>(c, data, ncomp, dir, kind);
        if (e == cudaSuccess) return fft_axis<T>(c, data, ncomp, 2, dir, kind);
        if (e != cudaErrorNotSupported) return e;
    } else {
        e = fft_axis<T>(c, data, ncomp, 2, dir, kind);
        if (e != cudaSuccess) return e;
        e = plane_xy<T>(c, data, ncomp, dir, kind);
        if (e != cudaErrorNotSupported) return e;
        e = fft_axis<T>(c, data, ncomp, 1, dir, kind);
        if (e != cudaSuccess) return e;
        return fft_axis<T>(c, data, ncomp, 0, dir, kind);
    }
    const int order_f[3] = {0, 1, 2}, order_i[3] = {2, 1, 0};
    const int* order = dir < 0 ? order_f : order_i;
    for (int q = 0; q < 3; ++q) {
        e = fft_axis<T>(c, data, ncomp, order[q], dir, kind);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// One spectral pass: forward x, y; fused z-forward / mode update / z-inverse;
// inverse y, x.
template <typename T>
cudaError_t spectral_pass(psatd_ctx* c, int mode, double scale) {
    const GridGeom g = geom(c);
    const Tables<T> tb = tables<T>(c);
    cplx<T>* f = static_cast<cplx<T>*>(c->fields);
    cudaError_t e;
    // the update fused into the x pass (N_x = 512, 1024) instead of the z pass: where the
    // z pass has no fused kernel; at N_x = 512, whose row kernel is the faster of the
    // two fused passes (512 x 256 x 256: 2.84 against 3.22 ms a step); and on planes of
    // 4 MB or more, where the z pass's 64-byte rows a plane apart reach 2.3 TB/s (1024 x
    // 512 x 256: 14.2 against 15.4 ms; 1024 x 256 x 256: 6.93 against 6.55 ms)
    const bool fused_z = g.Nz == 64 || g.Nz == 128 || g.Nz == 256;
    if (mode == KS_ROTATE && c->kernel_path == PSATD_PATH_AUTO && kspace_rows_supported(c->prec, g) &&
        (!fused_z || g.Nx == 512 || (long long)g.Nx * g.Ny >= 512 * 1024)) {
        // forward z, y; forward x, update, inverse x in one launch; inverse y, z
        if ((e = fft_axis<T>(c, f, 6, 2, -1, -1)) != cudaSuccess) return e;
        if ((e = fft_axis<T>(c, f, 6, 1, -1, -1)) != cudaSuccess) return e;
        e = timed(c, PSATD_KERNEL_KSPACE, [&] {
            ++c->launches;
            return launch_kspace_rows<T>(f, g, tb, c->stream);
        });
        if (e != cudaSuccess) return e;
        if ((e = fft_axis<T>(c, f, 6, 1, +1, -1)) != cudaSuccess) return e;
        return fft_axis<T>(c, f, 6, 2, +1, -1);
    }
    e = plane_xy<T>(c, f, 6, -1, -1);
    const bool fused_xy = (e == cudaSuccess);
    if (!fused_xy) {
        if (e != cudaErrorNotSupported) return e;
        if ((e = fft_axis<T>(c, f, 6, 0, -1, -1)) != cudaSuccess) return e;
        if ((e = fft_axis<T>(c, f, 6, 1, -1, -1)) != cudaSuccess) return e;
    }
    e = timed(c, PSATD_KERNEL_KSPACE, [&] {
        if (mode == KS_ROTATE && c->kernel_path == PSATD_PATH_AUTO && ensure_field_map(c)) {
            cudaError_t r = launch_kspace_tma<T>(c->field_map, f, g, tb, c->dev_err, c->stream);
            if (r != cudaErrorNotSupported) {
                ++c->launches;
                return r;
            }
        }
        // (the table is built on first use, outside graph capture; a capture before
        // that takes the generic projection below)
        if (mode == KS_PROJECT && c->kernel_path == PSATD_PATH_AUTO && (c->coef_proj.p || !capturing(c)) &&
            ensure_field_map(c)) {
            if (!c->coef_proj.p && upload_coef<T>(c, 0.0, &c->coef_proj, false, true) != PSATD_OK)
                return cudaErrorMemoryAllocation;
            Tables<T> tp = tb;
            tp.coef = static_cast<const ModeCoef<T>*>(c->coef_proj.p);
            cudaError_t r = launch_kspace_tma<T>(c->field_map, f, g, tp, c->dev_err, c->stream, false, true);
            if (r != cudaErrorNotSupported) {
                ++c->launches;
                return r;
            }
        }
        if (mode == KS_ROTATE && c->kernel_path != PSATD_PATH_GENERIC) {
            cudaError_t r = launch_kspace_fast<T>(f, g, tb, c->stream);
            if (r != cudaErrorNotSupported) {
                ++c->launches;
                return r;
            }
        }
        if (c->kernel_path != PSATD_PATH_GENERIC) {
            cudaError_t r = kspace_two<T>(f, g, tb, mode, scale, c->stream);
            if (r != cudaErrorNotSupported) {
                ++c->launches;
                return r;
            }
        }
        if (c->kernel_path != PSATD_PATH_GENERIC) {
            // a z length with register transforms but no fused kernel (1024 points in
            // float32; 512 have one in fft_two.cuh: step of 180 x 150 x 512 1.53 ms
            // with it, 1.68 ms with three launches): forward z, the per-mode update,
            // inverse z as three launches
            cudaError_t r = launch_fft_axis_fast<T>(f, 6, g, tb, 2, -1, c->stream);
            if (r != cudaErrorNotSupported) {
                ++c->launches;
                if (r != cudaSuccess) return r;
                if ((r = launch_modes<T>(f, g, tb, mode, scale, c->stream)) != cudaSuccess) return r;
                ++c->launches;
                r = launch_fft_axis_fast<T>(f, 6, g, tb, 2, +1, c->stream);
                ++c->launches;
                return r;
            }
        }
        return launch_kspace_z<T>(f, g, tb, mode, scale, c->stream, &c->launches);
    });
    if (e != cudaSuccess) return e;
    if (fused_xy) return plane_xy<T>(c, f, 6, +1, -1);
    if ((e = fft_axis<T>(c, f, 6, 1, +1, -1)) != cudaSuccess) return e;
    if ((e = fft_axis<T>(c, f, 6, 0, +1, -1)) != cudaSuccess) return e;
    return cudaSuccess;
}

// One real-field step: r2c plane transforms, the half-spectrum k-space pass
// (field slots and the x Nyquist array in one launch), c2r plane transforms.
// coef replaces the step's slot-ordered table (the projection, one step of T);
// project_b / project_e project B / E before the update (the one-time
// projection alone: B only, the update projects E; the projection followed by
// a step: both); spectral_out stops after the k-space pass, leaving the updated
// half spectrum in natural k_z order.
cudaError_t spectral_pass_real(psatd_ctx* c, const ModeCoef<float>* coef = nullptr, bool project_b = false,
                               bool spectral_out = false, bool project_e = false) {
    const GridGeom g = geom(c);
    const Tables<float> tb = tables<float>(c);
    float* f = static_cast<float*>(c->fields);
    float2* nyq = static_cast<float2*>(c->nyq.p);
    if (!ensure_field_map(c) || !c->nyq_map_ok) return cudaErrorNotSupported;
    cudaError_t e = timed(c, PSATD_KERNEL_PLANE_XY, [&] {
        ++c->launches;
        return launch_plane_rc(f, nyq, 6, g, tb, -1, c->stream);
    });
    if (e != cudaSuccess) return e;
    const HalfSlots<float> hs{static_cast<const float*>(c->slot_k.p),
                              coef ? coef : static_cast<const ModeCoef<float>*>(c->slot_coef.p), nyq, &c->nyq_map,
                              project_e};
    e = timed(c, PSATD_KERNEL_KSPACE, [&] {
        ++c->launches;
        return launch_kspace_tma<float>(c->field_map, reinterpret_cast<cplx<float>*>(f), g, tb, c->dev_err, c->stream,
                                        spectral_out, project_b, &hs);
    });
    if (e != cudaSuccess || spectral_out) return e;
    return timed(c, PSATD_KERNEL_PLANE_XY, [&] {
        ++c->launches;
        return launch_plane_rc(f, nyq, 6, g, tb, +1, c->stream);
    });
}

psatd_status upload_slot_tables(psatd_ctx* c) {
    const int nh = c->grid.Nx / 2;
    std::vector<float> k(nh);
    for (int p = 0; p < nh; ++p)
        k[p] = (float)(kTwoPi * (double)plane_rc_slot_mode(p) / (c->grid.Nx * c->grid.dx));
    CK(c, ensure_buf(c->slot_k, nh * sizeof(float)));
    CK(c, cudaMemcpy(c->slot_k.p, k.data(), nh * sizeof(float), cudaMemcpyHostToDevice));
    std::vector<int> mode(nh);
    for (int p = 0; p < nh; ++p) mode[p] = plane_rc_slot_mode(p);
    CK(c, ensure_buf(c->slot_mode, nh * sizeof(int)));
    CK(c, cudaMemcpy(c->slot_mode.p, mode.data(), nh * sizeof(int), cudaMemcpyHostToDevice));
    const size_t nn = (size_t)6 * c->grid.Ny * c->grid.Nz;
    CK(c, ensure_buf(c->nyq, nn * sizeof(float2)));
    CK(c, cudaMemset(c->nyq.p, 0, nn * sizeof(float2)));
    // 3D map {Ny, Nz, 6} of 8-byte elements, box {kspace_tma_box_x, Nz, 1}
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (enc && kspace_tma_box_z(c->grid.Nz)) {
        const cuuint64_t dims[3] = {(cuuint64_t)c->grid.Ny, (cuuint64_t)c->grid.Nz, 6};
        const cuuint64_t strides[2] = {(cuuint64_t)c->grid.Ny * 8, (cuuint64_t)c->grid.Ny * c->grid.Nz * 8};
        const cuuint32_t box[3] = {(cuuint32_t)kspace_tma_box_x(32), (cuuint32_t)kspace_tma_box_z(c->grid.Nz), 1};
        const cuuint32_t estr[3] = {1, 1, 1};
        c->nyq_map_ok = enc(&c->nyq_map, CU_TENSOR_MAP_DATA_TYPE_INT64, 3, c->nyq.p, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    return PSATD_OK;
}

double F_series(double t0) {
    const double t2 = t0 * t0;
    return t2 / 4 - t2 * t2 / 48 + t2 * t2 * t2 / 960;
}

}  // namespace

namespace {

// Forward x+y transform, then the k-space pass with the table of one step T that
// leaves the updated spectrum (with 1/N folded in) in storage.
template <typename T>
cudaError_t one_shot_spectrum(psatd_ctx* c, bool project_b) {
    const GridGeom g = geom(c);
    Tables<T> tb = tables<T>(c);
    tb.coef = static_cast<const ModeCoef<T>*>(c->coef_T.p);
    cplx<T>* f = static_cast<cplx<T>*>(c->fields);
    cudaError_t e = plane_xy<T>(c, f, 6, -1, -1);
    if (e == cudaErrorNotSupported) {
        if ((e = fft_axis<T>(c, f, 6, 0, -1, -1)) != cudaSuccess) return e;
        e = fft_axis<T>(c, f, 6, 1, -1, -1);
    }
    if (e != cudaSuccess) return e;
    return timed(c, PSATD_KERNEL_KSPACE, [&] {
        ++c->launches;
        if (c->kernel_path == PSATD_PATH_AUTO && ensure_field_map(c)) {
            cudaError_t r = launch_kspace_tma<T>(c->field_map, f, g, tb, c->dev_err, c->stream, true, project_b);
            if (r != cudaErrorNotSupported) return r;
        }
        if (c->kernel_path != PSATD_PATH_GENERIC) {
            cudaError_t r = kspace_two<T>(f, g, tb, project_b ? KS_ROTATE_SPECTRAL_PROJ : KS_ROTATE_SPECTRAL, 0.0,
                                          c->stream);
            if (r != cudaErrorNotSupported) return r;
        }
        --c->launches;
        return launch_kspace_z<T>(f, g, tb, project_b ? KS_ROTATE_SPECTRAL_PROJ : KS_ROTATE_SPECTRAL, 0.0,
                                  c->stream, &c->launches);
    });
}


// ---------------------------------------------------------------------------
// Persistent batched advance (multi_advance.cu)

bool same_plan(const AxisPlan& a, const AxisPlan& b) {
    if (a.N != b.N || a.npass != b.npass) return false;
    for (int i = 0; i < a.npass; ++i)
        if (a.radix[i] != b.radix[i]) return false;
    return true;
}

constexpr size_t kMultiHeader = 256;              // barrier counter at the start of the batch buffer
constexpr int kMultiMaxN = 1024;
constexpr unsigned long long kMultiWaitNs = 2000000000ull;   // 2 s per barrier wait

// tuned (radix schedule, tile-width scale) per (precision, axis length)
struct MultiChoice {
    int variant = 0, scale = 0;
    bool operator==(const MultiChoice& o) const { return variant == o.variant && scale == o.scale; }
};
std::map<std::pair<int, int>, MultiChoice> g_multi_tuned;
std::mutex g_multi_mutex;

MultiChoice multi_choice(int prec, int N) {
    std::lock_guard<std::mutex> lock(g_multi_mutex);
    auto it = g_multi_tuned.find({prec, N});
    return it == g_multi_tuned.end() ? MultiChoice{} : it->second;
}

// Tile width of the phase along `axis`: x rows (about 256 first-pass items per
// tile), y x-columns (128 contiguous bytes per row), z x-columns (64 bytes, six
// components held), scaled by 2^scale and halved until the tile fits; the column
// counts are powers of two.
template <typename T>
int multi_width(int axis, const psatd_grid& g, const AxisPlan& pl, int scale) {
    const int es = (int)sizeof(cplx<T>);
    const int N = axis_n(g, axis);
    int w = 1;
    if (axis == 0) w = std::max(1, std::min(128, 256 * pl.radix[0] / std::max(N, 1)));
    else
        while (w < g.Nx && w < (axis == 1 ? 128 : 64) / es) w *= 2;
    w = scale > 0 ? (w << scale) : (scale < 0 ? (w >> -scale) : w);
    w = std::max(1, std::min(w, axis == 0 ? 256 : 32));
    while (w > 1 && multi_tile_bytes<T>(axis, pl, w) > multi_tile_budget<T>()) w /= 2;
    return w;
}

struct MultiPrepared {
    const void* probs = nullptr;
    const long long* prefix = nullptr;
    unsigned* bar = nullptr;
    size_t tile = 0;
    long long max_items = 0;
};

// Describe the boxes (fields[p] replaces box p's storage when given), upload
// the descriptors to the lead context's buffer when they changed, and return
// the device pointers.  choice overrides the tuned schedules per axis length.
template <typename T>
psatd_status multi_prepare(psatd_ctx* const* ctxs, int n, const int* steps, void* const* fields,
                           const std::map<int, MultiChoice>* choice, MultiPrepared* out) {
    psatd_ctx* c0 = ctxs[0];
    std::vector<MultiProblem<T>> probs((size_t)n);
    std::vector<long long> prefix(3 * (size_t)(n + 1), 0);
    size_t tile = 0;
    for (int p = 0; p < n; ++p) {
        psatd_ctx* c = ctxs[p];
        MultiProblem<T>& P = probs[p];
        std::memset(&P, 0, sizeof P);
        P.f = static_cast<cplx<T>*>(fields ? fields[p] : c->fields);
        P.coef = static_cast<const ModeCoef<T>*>(c->coef.p);
        P.nsteps = steps[p];
        for (int a = 0; a < 3; ++a) {
            P.k[a] = static_cast<const T*>(c->k[a].p);
            P.N[a] = axis_n(c->grid, a);
            MultiChoice ch = multi_choice(c->prec, P.N[a]);
            if (choice) {
                auto it = choice->find(P.N[a]);
                if (it != choice->end()) ch = it->second;
            }
            make_plan_variant(P.N[a], ch.variant, &P.plan[a]);
            P.tp[a] = static_cast<const cplx<T>*>(c->twp[a].p) + c->twp_at[a][1 + (ch.variant & 1)];
            P.W[a] = multi_width<T>(a, c->grid, P.plan[a], ch.scale);
            // Compile-time tiles (16 uneven boxes: 9.45 ms against 11.2 ms with the
            // run-time passes): float32, two radices up to 16 and a tile within the
            // budget (z: 192 points; longer ones take the run-time passes at half the
            // width).  They have widths of their own, so a tuned width (scale) keeps the
            // run-time passes too.
            P.two[a] = -1;
            if (sizeof(T) == 4 && ch.scale == 0) {
                const int own = a == 0 ? two_rows_per_tile(P.plan[a]) : (a == 1 ? 16 : 8);
                const int id = two_pair_index(P.plan[a]);
                if (id >= 0 && multi_tile_bytes<T>(a, P.plan[a], own) <= multi_tile_budget<T>()) {
                    P.two[a] = id;
                    P.W[a] = own;
                }
            }
            tile = std::max(tile, multi_tile_bytes<T>(a, P.plan[a], P.W[a]));
        }
        const long long Nx = P.N[0], Ny = P.N[1], Nz = P.N[2];
        const long long items[3] = {(6 * Nz * Ny + P.W[0] - 1) / P.W[0], 6 * Nz * ((Nx + P.W[1] - 1) / P.W[1]),
                                    Ny * ((Nx + P.W[2] - 1) / P.W[2])};
        for (int a = 0; a < 3; ++a) prefix[a * (n + 1) + p + 1] = prefix[a * (n + 1) + p] + items[a];
    }
    long long max_items = 0;
    for (int a = 0; a < 3; ++a) max_items = std::max(max_items, prefix[a * (n + 1) + n]);
    const size_t pbytes = (prefix.size() * sizeof(long long) + 15) / 16 * 16;
    const size_t dbytes = probs.size() * sizeof(MultiProblem<T>);
    std::vector<unsigned char> sig(pbytes + dbytes, 0);
    std::memcpy(sig.data(), prefix.data(), prefix.size() * sizeof(long long));
    std::memcpy(sig.data() + pbytes, probs.data(), dbytes);
    if (c0->multi.bytes < kMultiHeader + sig.size() || sig != c0->multi_sig) {
        if (capturing(c0))
            return fail(c0, PSATD_ERR_STATE, "inside a batch capture psatd_multi_advance needs the boxes, step counts "
                                             "and tuning of a call made before the capture");
        c0->multi_sig.clear();
        CK(c0, cudaStreamSynchronize(c0->stream));           // a launch in flight may still read the buffer
        CK(c0, ensure_buf(c0->multi, kMultiHeader + sig.size()));
        CK(c0, cudaMemcpyAsync(static_cast<char*>(c0->multi.p) + kMultiHeader, sig.data(), sig.size(),
                               cudaMemcpyHostToDevice, c0->stream));
        CK(c0, cudaStreamSynchronize(c0->stream));
        c0->multi_sig = std::move(sig);
    }
    char* base = static_cast<char*>(c0->multi.p);
    out->bar = reinterpret_cast<unsigned*>(base);
    out->prefix = reinterpret_cast<const long long*>(base + kMultiHeader);
    out->probs = base + kMultiHeader + pbytes;
    out->tile = tile;
    out->max_items = max_items;
    return PSATD_OK;
}

template <typename T>
psatd_status multi_launch(psatd_ctx* const* ctxs, int n, int nsteps, const MultiPrepared& m,
                          unsigned long long limit_ns, unsigned extra) {
    psatd_ctx* c0 = ctxs[0];
    nvtxRangePushA("multi_advance");
    cudaError_t e = launch_multi_advance<T>(static_cast<const MultiProblem<T>*>(m.probs), m.prefix, n, nsteps, m.tile,
                                            m.max_items, m.bar, c0->dev_err, limit_ns, extra, c0->stream, nullptr);
    nvtxRangePop();
    if (e != cudaSuccess) return cuda_fail(c0, e, "persistent batched advance launch");
    ++c0->launches;
    return PSATD_OK;
}

// Argument checks shared by the batched entry points; errors go to ctxs[0].
psatd_status multi_check(psatd_ctx* const* ctxs, int n) {
    if (!ctxs || n < 1) return fail(nullptr, PSATD_ERR_ARG, "need at least one context");
    for (int p = 0; p < n; ++p)
        if (!ctxs[p]) return fail(nullptr, PSATD_ERR_ARG, "NULL context in the list");
    psatd_ctx* c0 = ctxs[0];
    std::vector<const void*> seen;
    for (int p = 0; p < n; ++p) {
        psatd_ctx* c = ctxs[p];
        psatd_status st = check_ctx(c, true, true);
        if (st) return fail(c0, st, "context " + std::to_string(p) + ": " + c->err);
        if (c->real_fields) return fail(c0, PSATD_ERR_STATE, "the batched advance needs complex field storage");
        if (c->prec != c0->prec) return fail(c0, PSATD_ERR_ARG, "all contexts need the same precision");
        if (c->stream != c0->stream || c->device != c0->device)
            return fail(c0, PSATD_ERR_ARG, "all contexts need the same device and stream");
        for (int a = 0; a < 3; ++a)
            if (axis_n(c->grid, a) > kMultiMaxN)
                return fail(c0, PSATD_ERR_SIZE, "the batched advance takes axis lengths up to 1024");
        seen.push_back(c->fields);
    }
    std::sort(seen.begin(), seen.end());
    if (std::adjacent_find(seen.begin(), seen.end()) != seen.end())
        return fail(c0, PSATD_ERR_ARG, "two contexts share field storage");
    return check_ctx(c0, true, true);
}

}  // namespace

extern "C" {

const char* psatd_status_string(psatd_status s) {
    switch (s) {
        case PSATD_OK: return "PSATD_OK";
        case PSATD_ERR_ARG: return "PSATD_ERR_ARG";
        case PSATD_ERR_SIZE: return "PSATD_ERR_SIZE";
        case PSATD_ERR_OOM: return "PSATD_ERR_OOM";
        case PSATD_ERR_CUDA: return "PSATD_ERR_CUDA";
        case PSATD_ERR_TIMEOUT: return "PSATD_ERR_TIMEOUT";
        case PSATD_ERR_STATE: return "PSATD_ERR_STATE";
    }
    return "PSATD_ERR_UNKNOWN";
}

const char* psatd_last_error(const psatd_ctx* ctx) {
    return ctx ? ctx->err.c_str() : g_create_error.c_str();
}

double psatd_d_min(double R0, double L, double theta) {
    const double rmin = R0 - 0.5 * L, rmax = R0 + 0.5 * L;
    const double s = rmin * std::sin(theta);
    return -rmin * std::cos(theta) + std::sqrt(rmax * rmax - s * s);
}

psatd_status psatd_init_grid(const psatd_grid* grid, const psatd_mapping* mapping, double dt,
                             int precision, void* cuda_stream, int flags, psatd_ctx** out) {
    if (!grid || !out) return fail(nullptr, PSATD_ERR_ARG, "NULL grid or out pointer");
    *out = nullptr;
    if (precision != 32 && precision != 64) return fail(nullptr, PSATD_ERR_ARG, "precision must be 32 or 64");
    const int Ns[3] = {grid->Nx, grid->Ny, grid->Nz};
    for (int a = 0; a < 3; ++a) {
        AxisPlan p;
        if (Ns[a] < 1 || Ns[a] > kMaxN || !make_plan(Ns[a], &p)) {
            char b[160];
            snprintf(b, sizeof b, "axis %d: N=%d must be in 1..%d with prime factors 2, 3, 5 only", a, Ns[a], kMaxN);
            return fail(nullptr, PSATD_ERR_SIZE, b);
        }
    }
    const double ds[3] = {grid->dx, grid->dy, grid->dz};
    for (double d : ds)
        if (!(is_finite(d) && d > 0)) return fail(nullptr, PSATD_ERR_ARG, "dx, dy, dz must be finite and > 0");
    if (!(is_finite(grid->c) && grid->c > 0)) return fail(nullptr, PSATD_ERR_ARG, "c must be finite and > 0");
    if (!is_finite(grid->x_min) || !is_finite(grid->y_min) || !is_finite(grid->z_min))
        return fail(nullptr, PSATD_ERR_ARG, "x_min, y_min, z_min must be finite");
    if (!is_finite(dt)) return fail(nullptr, PSATD_ERR_ARG, "dt must be finite");
    if (mapping && !(is_finite(mapping->R0) && is_finite(mapping->L) && mapping->L >= 0))
        return fail(nullptr, PSATD_ERR_ARG, "mapping R0, L must be finite, L >= 0");
    const bool real = (flags & PSATD_FLAG_REAL_FIELDS) != 0;
    if (real && !(precision == 32 && grid->Nx == 256 && grid->Ny == 256 &&
                  (grid->Nz == 64 || grid->Nz == 128 || grid->Nz == 256)))
        return fail(nullptr, PSATD_ERR_ARG, "real fields need precision 32 and a 256 x 256 x {64, 128, 256} grid");

    psatd_ctx* c = new (std::nothrow) psatd_ctx();
    if (!c) return fail(nullptr, PSATD_ERR_OOM, "host allocation failed");
    c->grid = *grid;
    if (mapping) c->mapping = *mapping;
    c->dt = dt;
    c->prec = precision;
    c->real_fields = real;
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    for (int a = 0; a < 3; ++a) context_plan(Ns[a], precision, a, &c->plan[a]);

    cudaError_t e = cudaGetDevice(&c->device);
    psatd_status st = PSATD_OK;
    if (e != cudaSuccess) st = cuda_fail(c, e, "cudaGetDevice");
    if (st == PSATD_OK) st = precision == 64 ? upload_axis_tables<double>(c) : upload_axis_tables<float>(c);
    if (st == PSATD_OK && real) st = upload_slot_tables(c);
    if (st == PSATD_OK) st = set_coef(c, dt);
    if (st == PSATD_OK) {
        e = lib_malloc(reinterpret_cast<void**>(&c->dev_err), sizeof(int));
        if (e == cudaSuccess) e = cudaMemset(c->dev_err, 0, sizeof(int));
        if (e != cudaSuccess) st = cuda_fail(c, e, "cudaMalloc(error word)");
    }
    if (st == PSATD_OK && !(flags & PSATD_FLAG_NO_FIELD_ALLOC)) {
        const size_t bytes = 6 * n_cells(*grid) * value_size(c);
        e = lib_malloc(&c->fields, bytes);
        if (e != cudaSuccess) {
            c->fields = nullptr;
            st = cuda_fail(c, e, "cudaMalloc(fields)");
        } else {
            c->field_bytes = bytes;
            c->own_fields = true;
            e = cudaMemsetAsync(c->fields, 0, bytes, c->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
            if (e != cudaSuccess) st = cuda_fail(c, e, "cudaMemset(fields)");
        }
    }
    if (st != PSATD_OK) {
        g_create_error = c->err;
        psatd_destroy(c);
        return st;
    }
    *out = c;
    return PSATD_OK;
}

void psatd_destroy(psatd_ctx* c) {
    if (!c) return;
    cudaSetDevice(c->device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    else cudaDeviceSynchronize();
    if (c->own_fields && c->fields) lib_free(c->fields);
    if (c->dev_err) lib_free(c->dev_err);
    for (int a = 0; a < 3; ++a) { free_buf(c->tw[a]); free_buf(c->k[a]); free_buf(c->twp[a]); }
    free_buf(c->coef);
    free_buf(c->coef_T);
    free_buf(c->coef_proj);
    free_buf(c->slot_k); free_buf(c->slot_coef); free_buf(c->nyq);
    free_buf(c->slot_mode); free_buf(c->slot_coef_proj);
    for (int a = 0; a < 3; ++a) free_buf(c->tw2[a]);
    free_buf(c->diag_spec); free_buf(c->diag_partial); free_buf(c->diag_out); free_buf(c->diag_nyq);
    free_buf(c->lprof);
    free_buf(c->multi);
    free_buf(c->samp_wx); free_buf(c->samp_wy); free_buf(c->samp_wz);
    free_buf(c->samp_g); free_buf(c->samp_h); free_buf(c->samp_out);
    for (auto& p : c->pending) { c->ev_pool.push_back(p.a); c->ev_pool.push_back(p.b); }
    for (cudaEvent_t e : c->ev_pool) cudaEventDestroy(e);
    delete c;
}

psatd_status psatd_set_dt(psatd_ctx* c, double dt) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "not allowed while a batch is being captured");
    if (!is_finite(dt)) return fail(c, PSATD_ERR_ARG, "dt must be finite");
    st = set_coef(c, dt);
    if (st == PSATD_OK) c->dt = dt;
    return st;
}

psatd_status psatd_set_pulse_profile(psatd_ctx* c, const double* samples, int n, double zeta0, double dzeta) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    if (!samples) return fail(c, PSATD_ERR_ARG, "NULL profile samples");
    if (n < 2 || n > (1 << 20)) return fail(c, PSATD_ERR_ARG, "profile needs 2 <= n <= 1048576 samples");
    if (!is_finite(zeta0) || !is_finite(dzeta) || !(dzeta > 0))
        return fail(c, PSATD_ERR_ARG, "profile needs finite zeta0 and dzeta > 0");
    for (int i = 0; i < 2 * n; ++i)
        if (!is_finite(samples[i])) return fail(c, PSATD_ERR_ARG, "profile samples must be finite");
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "psatd_set_pulse_profile cannot be captured in a batch");
    CK(c, cudaStreamSynchronize(c->stream));           // a previous table may still be read
    CK(c, ensure_buf(c->lprof, (size_t)n * sizeof(double2)));
    CK(c, cudaMemcpy(c->lprof.p, samples, (size_t)n * sizeof(double2), cudaMemcpyHostToDevice));
    c->lprof_n = n;
    c->lprof_z0 = zeta0;
    c->lprof_dz = dzeta;
    return PSATD_OK;
}

psatd_status psatd_set_mapping(psatd_ctx* c, const psatd_mapping* m) {
    if (!c || !m) return fail(c, PSATD_ERR_ARG, "NULL argument");
    if (!(is_finite(m->R0) && is_finite(m->L) && m->L >= 0)) return fail(c, PSATD_ERR_ARG, "mapping R0, L must be finite, L >= 0");
    c->mapping = *m;
    return PSATD_OK;
}

psatd_status psatd_bind_fields(psatd_ctx* c, void* dev_ptr, size_t bytes) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    const size_t need = 6 * n_cells(c->grid) * value_size(c);
    if (!dev_ptr) return fail(c, PSATD_ERR_ARG, "NULL field pointer");
    if (bytes < need) return fail(c, PSATD_ERR_ARG, "field storage too small");
    if (reinterpret_cast<uintptr_t>(dev_ptr) % 256 != 0) return fail(c, PSATD_ERR_ARG, "field storage must be 256-byte aligned");
    cudaPointerAttributes at;
    cudaError_t e = cudaPointerGetAttributes(&at, dev_ptr);
    if (e != cudaSuccess) return cuda_fail(c, e, "cudaPointerGetAttributes");
    if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)
        return fail(c, PSATD_ERR_ARG, "field storage must be device memory");
    if (c->own_fields && c->fields) {
        CK(c, cudaStreamSynchronize(c->stream));
        lib_free(c->fields);
    }
    c->fields = dev_ptr;
    c->field_bytes = bytes;
    c->own_fields = false;
    return PSATD_OK;
}

psatd_status psatd_fields(psatd_ctx* c, void** dev_ptr, size_t* bytes) {
    if (!c || !dev_ptr) return fail(c, PSATD_ERR_ARG, "NULL argument");
    *dev_ptr = c->fields;
    if (bytes) *bytes = c->field_bytes;
    return PSATD_OK;
}

static psatd_status copy_field(psatd_ctx* c, int comp, void* dst, const void* src, int on_device,
                               bool to_lib) {
    psatd_status st = check_ctx(c, true);
    if (st) return st;
    if (comp < -1 || comp > 5) return fail(c, PSATD_ERR_ARG, "comp must be -1..5");
    if (!on_device && capturing(c)) return fail(c, PSATD_ERR_STATE, "host copies are not allowed while a batch is being captured");
    if (!(to_lib ? src : dst)) return fail(c, PSATD_ERR_ARG, "NULL buffer");
    const size_t per = n_cells(c->grid) * value_size(c);
    const size_t bytes = comp < 0 ? 6 * per : per;
    char* lib = static_cast<char*>(c->fields) + (comp < 0 ? 0 : comp * per);
    cudaMemcpyKind kind;
    if (to_lib) kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    else kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    CK(c, cudaMemcpyAsync(to_lib ? lib : dst, to_lib ? src : lib, bytes, kind, c->stream));
    if (!on_device) CK(c, cudaStreamSynchronize(c->stream));
    if (!to_lib && !on_device) return check_device_error(c);
    return PSATD_OK;
}

psatd_status psatd_set_field(psatd_ctx* c, int comp, const void* src, int src_on_device) {
    psatd_status st = copy_field(c, comp, nullptr, src, src_on_device, true);
    if (st == PSATD_OK && comp < 0) c->holds_spectrum = false;
    return st;
}

psatd_status psatd_get_field(psatd_ctx* c, int comp, void* dst, int dst_on_device) {
    return copy_field(c, comp, dst, nullptr, dst_on_device, false);
}

psatd_status psatd_init_pulse(psatd_ctx* c, const psatd_pulse* p) {
    psatd_status st = check_ctx(c, true);
    if (st) return st;
    if (!p) return fail(c, PSATD_ERR_ARG, "NULL pulse");
    if (p->kind != PSATD_PULSE_FLAT_TOP && p->kind != PSATD_PULSE_GAUSSIAN && p->kind != PSATD_PULSE_PROFILE)
        return fail(c, PSATD_ERR_ARG, "unknown pulse kind");
    if (p->kind == PSATD_PULSE_PROFILE && c->lprof_n < 2)
        return fail(c, PSATD_ERR_STATE, "a profile pulse needs psatd_set_pulse_profile first");
    const double vals[8] = {p->lambda, p->theta, p->eps, p->P0, p->n_cycles, p->cep, p->ellipticity, p->pol_angle};
    for (double v : vals)
        if (!is_finite(v)) return fail(c, PSATD_ERR_ARG, "pulse parameters must be finite");
    if (!(p->lambda > 0) || !(p->theta > 0) || p->eps < 0 || p->P0 < 0)
        return fail(c, PSATD_ERR_ARG, "need lambda > 0, theta > 0, eps >= 0, P0 >= 0");
    if (p->kind == PSATD_PULSE_GAUSSIAN && !(p->n_cycles > 0))
        return fail(c, PSATD_ERR_ARG, "Gaussian pulse needs n_cycles > 0");
    if (!(c->mapping.R0 > 0) || !(c->mapping.L > 0))
        return fail(c, PSATD_ERR_ARG, "mapping R0 and L must be > 0 for a pulse");
    if (p->kind != PSATD_PULSE_GAUSSIAN && !(std::cos(p->theta) < 1.0))
        return fail(c, PSATD_ERR_ARG, "flat-top theta too small");

    PulseParams pp;
    pp.kind = p->kind; pp.div_project = p->div_project;
    pp.lambda = p->lambda; pp.theta = p->theta; pp.eps = p->eps; pp.P0 = p->P0;
    pp.n_cycles = p->n_cycles; pp.cep = p->cep; pp.ellipticity = p->ellipticity;
    pp.pol_angle = p->pol_angle;
    pp.prof = static_cast<const double2*>(c->lprof.p);
    pp.prof_n = c->lprof_n;
    pp.prof_z0 = c->lprof_z0;
    pp.prof_dz = c->lprof_dz;
    if (p->kind != PSATD_PULSE_GAUSSIAN)
        pp.amp = std::sqrt(4.0 * p->P0 / (c->grid.c * (1.0 - std::cos(p->theta))));           // Eq. 9
    else
        pp.amp = std::sqrt(4.0 * p->P0 / (c->grid.c * c->mapping.R0 * c->mapping.R0 * F_series(p->theta)));

    // replicas m whose copy x~ + m D can meet the shell |R| <= R_max
    const double D = c->grid.Nx * c->grid.dx;
    const double rmax = c->mapping.R0 + 0.5 * c->mapping.L;
    const int m_lo = (int)std::floor((-rmax - (c->grid.x_min + D)) / D) - 1;
    const int m_hi = (int)std::ceil((rmax - c->grid.x_min) / D) + 1;
    if (m_hi - m_lo > 100000) return fail(c, PSATD_ERR_ARG, "shell spans too many replicas of the layer");

    ShellGeom sh{c->mapping.R0, c->mapping.L};
    const GridGeom g = geom(c);
    cudaError_t e = timed(c, PSATD_KERNEL_INIT, [&] {
        if (c->real_fields)                            // the pulse is real: written straight into real storage
            return launch_init_pulse_real(static_cast<float*>(c->fields), g, sh, pp, m_lo, m_hi, c->stream, &c->launches);
        return c->prec == 64
            ? launch_init_pulse<double>(static_cast<cplx<double>*>(c->fields), g, sh, pp, m_lo, m_hi, c->stream, &c->launches)
            : launch_init_pulse<float>(static_cast<cplx<float>*>(c->fields), g, sh, pp, m_lo, m_hi, c->stream, &c->launches);
    });
    if (e != cudaSuccess) return cuda_fail(c, e, "init_pulse launch");
    c->holds_spectrum = false;
    if (p->div_project && c->real_fields) {
        // the projection as one real-field pass with C = 1/Ntot, S = 0 and B projected
        if (!c->slot_coef_proj.p) {
            if (capturing(c)) return fail(c, PSATD_ERR_STATE, "the first projection cannot run inside a batch capture");
            st = upload_coef<float>(c, 0.0, &c->slot_coef_proj, true, true);
            if (st) return st;
        }
        e = spectral_pass_real(c, static_cast<const ModeCoef<float>*>(c->slot_coef_proj.p), true, false);
        if (e != cudaSuccess) return cuda_fail(c, e, "projection launch");
    } else if (p->div_project) {
        const double scale = 1.0 / (double)n_cells(c->grid);
        e = c->prec == 64 ? spectral_pass<double>(c, KS_PROJECT, scale) : spectral_pass<float>(c, KS_PROJECT, scale);
        if (e != cudaSuccess) return cuda_fail(c, e, "projection launch");
    }
    c->t = 0.0;
    return PSATD_OK;
}



psatd_status psatd_advance(psatd_ctx* c, int n_steps) {
    psatd_status st = check_ctx(c, true, true);
    if (st) return st;
    if (n_steps < 0) return fail(c, PSATD_ERR_ARG, "n_steps must be >= 0");
    psatd_batch* b = capturing(c);
    if (b && c->prof_on) return fail(c, PSATD_ERR_STATE, "profiling must be off while capturing a batch");
    for (int s = 0; s < n_steps; ++s) {
        cudaError_t e = inject_due() ? (cudaError_t)g_inject_error.load()
                        : c->real_fields ? spectral_pass_real(c)
                        : c->prec == 64 ? spectral_pass<double>(c, KS_ROTATE, 0.0)
                                        : spectral_pass<float>(c, KS_ROTATE, 0.0);
        if (e != cudaSuccess) return cuda_fail(c, e, "advance launch");
        if (!b) c->t += c->dt;
    }
    if (b) b->time_advance.push_back({c, n_steps * c->dt});
    return PSATD_OK;
}

psatd_status psatd_fft(psatd_ctx* c, int direction) {
    psatd_status st = check_ctx(c, true, true);
    if (st) return st;
    if (direction != PSATD_FORWARD && direction != PSATD_INVERSE)
        return fail(c, PSATD_ERR_ARG, "direction must be PSATD_FORWARD or PSATD_INVERSE");
    if (c->real_fields) return fail(c, PSATD_ERR_STATE, "psatd_fft works on complex field storage only");
    cudaError_t e = c->prec == 64 ? fft3d<double>(c, static_cast<cplx<double>*>(c->fields), 6, direction)
                                  : fft3d<float>(c, static_cast<cplx<float>*>(c->fields), 6, direction);
    if (e != cudaSuccess) return cuda_fail(c, e, "fft launch");
    return PSATD_OK;
}

psatd_status psatd_sample_focal_plane(psatd_ctx* c, double x_phys, int ny, int nz, double y0, double y1,
                                      double z0, double z1, int comp_mask, void* dst, int dst_on_device) {
    psatd_status st = check_ctx(c, true);
    if (st) return st;
    if (!dst) return fail(c, PSATD_ERR_ARG, "NULL dst");
    if (ny < 1 || nz < 1 || ny > 4096 || nz > 4096) return fail(c, PSATD_ERR_ARG, "ny, nz must be 1..4096");
    if (!(is_finite(x_phys) && is_finite(y0) && is_finite(y1) && is_finite(z0) && is_finite(z1)))
        return fail(c, PSATD_ERR_ARG, "plane coordinates must be finite");
    if (comp_mask <= 0 || comp_mask > 63) return fail(c, PSATD_ERR_ARG, "comp_mask must select 1..6 components");
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "sample_focal_plane is not captured into batches; use psatd_focal_one_shot");
    int comps[6], nc = 0;
    for (int a = 0; a < 6; ++a)
        if (comp_mask & (1 << a)) comps[nc++] = a;
    const psatd_grid& g = c->grid;
    CK(c, ensure_buf(c->samp_wx, g.Nx * sizeof(double2)));
    CK(c, ensure_buf(c->samp_wy, (size_t)ny * g.Ny * sizeof(double2)));
    CK(c, ensure_buf(c->samp_wz, (size_t)nz * g.Nz * sizeof(double2)));
    CK(c, ensure_buf(c->samp_g, (size_t)nc * g.Nz * g.Ny * sizeof(double2)));
    CK(c, ensure_buf(c->samp_h, (size_t)nc * g.Nz * ny * sizeof(double2)));
    const size_t out_bytes = (size_t)nc * nz * ny * cplx_size(c->prec);
    void* out = dst;
    if (!dst_on_device) {
        CK(c, ensure_buf(c->samp_out, out_bytes));
        out = c->samp_out.p;
    }
    SampleScratch sc{static_cast<double2*>(c->samp_wx.p), static_cast<double2*>(c->samp_wy.p),
                     static_cast<double2*>(c->samp_wz.p), static_cast<double2*>(c->samp_g.p),
                     static_cast<double2*>(c->samp_h.p)};
    ShellGeom sh{c->mapping.R0, c->mapping.L};
    const GridGeom gg = geom(c);
    cudaError_t e = timed(c, PSATD_KERNEL_SAMPLE, [&] {
        if (c->real_fields)
            return launch_sample_plane_real(static_cast<const float*>(c->fields), static_cast<const float2*>(c->nyq.p), static_cast<const int*>(c->slot_mode.p), gg, sh, x_phys, ny, nz, y0, y1, z0, z1, c->t, comps, nc, sc, static_cast<float2*>(out), c->stream, &c->launches, c->holds_spectrum);
        return c->prec == 64
            ? launch_sample_plane<double>(static_cast<const cplx<double>*>(c->fields), gg, sh, x_phys, ny, nz, y0, y1, z0, z1, c->t, comps, nc, sc, static_cast<cplx<double>*>(out), c->stream, &c->launches, c->holds_spectrum)
            : launch_sample_plane<float>(static_cast<const cplx<float>*>(c->fields), gg, sh, x_phys, ny, nz, y0, y1, z0, z1, c->t, comps, nc, sc, static_cast<cplx<float>*>(out), c->stream, &c->launches, c->holds_spectrum);
    });
    if (e != cudaSuccess) return cuda_fail(c, e, "sample launch");
    if (!dst_on_device) {
        CK(c, cudaMemcpyAsync(dst, out, out_bytes, cudaMemcpyDeviceToHost, c->stream));
        CK(c, cudaStreamSynchronize(c->stream));
        return check_device_error(c);
    }
    return PSATD_OK;
}

psatd_status psatd_focal_one_shot(psatd_ctx* c, const psatd_pulse* pulse, double T, double x_phys, int ny,
                                  int nz, double y0, double y1, double z0, double z1, int comp_mask, void* dst,
                                  int dst_on_device) {
    psatd_status st = check_ctx(c, true);
    if (st) return st;
    if (!is_finite(T)) return fail(c, PSATD_ERR_ARG, "T must be finite");
    if (!dst) return fail(c, PSATD_ERR_ARG, "NULL dst");
    if (ny < 1 || nz < 1 || ny > 4096 || nz > 4096) return fail(c, PSATD_ERR_ARG, "ny, nz must be 1..4096");
    if (comp_mask <= 0 || comp_mask > 63) return fail(c, PSATD_ERR_ARG, "comp_mask must select 1..6 components");
    if (!(is_finite(x_phys) && is_finite(y0) && is_finite(y1) && is_finite(z0) && is_finite(z1)))
        return fail(c, PSATD_ERR_ARG, "plane coordinates must be finite");
    psatd_batch* cap = capturing(c);
    if (cap) {
        const psatd_grid& g0 = c->grid;
        int nc0 = 0;
        for (int a = 0; a < 6; ++a) nc0 += (comp_mask >> a) & 1;
        const bool ready = c->coef_T_ok && c->coef_T_step == T && dst_on_device && !c->prof_on &&
                           c->samp_wy.bytes >= (size_t)ny * g0.Ny * sizeof(double2) &&
                           c->samp_wz.bytes >= (size_t)nz * g0.Nz * sizeof(double2) &&
                           c->samp_g.bytes >= (size_t)nc0 * g0.Nz * g0.Ny * sizeof(double2) &&
                           c->samp_h.bytes >= (size_t)nc0 * g0.Nz * ny * sizeof(double2) && c->samp_wx.p;
        if (!ready)
            return fail(c, PSATD_ERR_STATE, "inside a batch capture the same one-shot (T, plane size, device "
                                            "dst) must have run once before, with profiling off");
    }
    if (!c->coef_T_ok || c->coef_T_step != T) {
        // real fields: the table in the slot order of the half spectrum (the pulse
        // initialisation below is an ordinary launch between it and its reader)
        c->coef_T_ok = false;
        st = c->prec == 64 ? upload_coef<double>(c, T, &c->coef_T, false, false, false)
                           : upload_coef<float>(c, T, &c->coef_T, c->real_fields, false, false);
        if (st) return st;
        c->coef_T_ok = true;
        c->coef_T_step = T;
    }
    psatd_pulse p = *pulse;
    const int project = p.div_project;
    p.div_project = 0;
    st = psatd_init_pulse(c, &p);
    if (st) return st;
    cudaError_t e = c->real_fields ? spectral_pass_real(c, static_cast<const ModeCoef<float>*>(c->coef_T.p),
                                                        project != 0, true, project != 0)
                    : c->prec == 64 ? one_shot_spectrum<double>(c, project != 0)
                                    : one_shot_spectrum<float>(c, project != 0);
    if (e != cudaSuccess) return cuda_fail(c, e, "one-shot launch");
    c->holds_spectrum = true;
    c->t = T;
    if (cap) cap->time_set.push_back({c, T});
    int comps[6], nc = 0;
    for (int a = 0; a < 6; ++a)
        if (comp_mask & (1 << a)) comps[nc++] = a;
    const psatd_grid& g = c->grid;
    CK(c, ensure_buf(c->samp_wx, g.Nx * sizeof(double2)));
    CK(c, ensure_buf(c->samp_wy, (size_t)ny * g.Ny * sizeof(double2)));
    CK(c, ensure_buf(c->samp_wz, (size_t)nz * g.Nz * sizeof(double2)));
    CK(c, ensure_buf(c->samp_g, (size_t)nc * g.Nz * g.Ny * sizeof(double2)));
    CK(c, ensure_buf(c->samp_h, (size_t)nc * g.Nz * ny * sizeof(double2)));
    const size_t out_bytes = (size_t)nc * nz * ny * cplx_size(c->prec);
    void* out = dst;
    if (!dst_on_device) {
        CK(c, ensure_buf(c->samp_out, out_bytes));
        out = c->samp_out.p;
    }
    SampleScratch sc{static_cast<double2*>(c->samp_wx.p), static_cast<double2*>(c->samp_wy.p),
                     static_cast<double2*>(c->samp_wz.p), static_cast<double2*>(c->samp_g.p),
                     static_cast<double2*>(c->samp_h.p)};
    ShellGeom sh{c->mapping.R0, c->mapping.L};
    const GridGeom gg = geom(c);
    e = timed(c, PSATD_KERNEL_SAMPLE, [&] {
        if (c->real_fields)
            return launch_sample_plane_real(static_cast<const float*>(c->fields), static_cast<const float2*>(c->nyq.p), static_cast<const int*>(c->slot_mode.p), gg, sh, x_phys, ny, nz, y0, y1, z0, z1, T, comps, nc, sc, static_cast<float2*>(out), c->stream, &c->launches, true);
        return c->prec == 64
            ? launch_sample_plane<double>(static_cast<const cplx<double>*>(c->fields), gg, sh, x_phys, ny, nz, y0, y1, z0, z1, T, comps, nc, sc, static_cast<cplx<double>*>(out), c->stream, &c->launches, true)
            : launch_sample_plane<float>(static_cast<const cplx<float>*>(c->fields), gg, sh, x_phys, ny, nz, y0, y1, z0, z1, T, comps, nc, sc, static_cast<cplx<float>*>(out), c->stream, &c->launches, true);
    });
    if (e != cudaSuccess) return cuda_fail(c, e, "one-shot sample launch");
    if (!dst_on_device) {
        CK(c, cudaMemcpyAsync(dst, out, out_bytes, cudaMemcpyDeviceToHost, c->stream));
        CK(c, cudaStreamSynchronize(c->stream));
        return check_device_error(c);
    }
    return PSATD_OK;
}

namespace {

// Diagnostics of real float32 storage without a complex copy: the energy from
// the real fields; per field (E, then B) its three components copied to a real
// scratch, taken to the half spectrum by the real-field plane kernel and the z
// transform of the slots and of the x-Nyquist array, and the divergence maxima
// over the stored modes.
psatd_status diagnostics_real(psatd_ctx* c, double host[6]) {
    const GridGeom g = geom(c);
    const Tables<float> tb = tables<float>(c);
    const size_t n = n_cells(c->grid);
    const size_t nq = (size_t)3 * c->grid.Nz * c->grid.Ny;
    CK(c, ensure_buf(c->diag_spec, 3 * n * sizeof(float)));
    CK(c, ensure_buf(c->diag_nyq, nq * sizeof(float2)));
    CK(c, ensure_buf(c->diag_partial, (size_t)kDiagBlocks * 2 * sizeof(double)));
    CK(c, ensure_buf(c->diag_out, 8 * sizeof(double)));
    double* partial = static_cast<double*>(c->diag_partial.p);
    double* res = static_cast<double*>(c->diag_out.p);
    float* spec = static_cast<float*>(c->diag_spec.p);
    float2* nyq = static_cast<float2*>(c->diag_nyq.p);
    cudaError_t e = timed(c, PSATD_KERNEL_DIAG, [&] {
        cudaError_t r = launch_energy_real(static_cast<const float*>(c->fields), n, partial, kDiagBlocks, c->stream,
                                           &c->launches);
        if (r != cudaSuccess) return r;
        return launch_reduce_final(partial, kDiagBlocks, 2, 2, res, c->stream, &c->launches);
    });
    if (e != cudaSuccess) return cuda_fail(c, e, "energy launch");
    GridGeom gs = g, gq = g;                          // the slots, the x-Nyquist array as complex grids
    gs.Nx = g.Nx / 2;
    gq.Nx = g.Ny;
    gq.Ny = 1;
    for (int half = 0; half < 2; ++half) {
        CK(c, cudaMemcpyAsync(spec, static_cast<const float*>(c->fields) + (size_t)3 * half * n, 3 * n * sizeof(float),
                              cudaMemcpyDeviceToDevice, c->stream));
        e = timed(c, PSATD_KERNEL_DIAG, [&] {
            c->launches += 4;
            cudaError_t r = launch_plane_rc(spec, nyq, 3, g, tb, -1, c->stream);
            if (r == cudaSuccess)
                r = launch_fft_axis_fast<float>(reinterpret_cast<cplx<float>*>(spec), 3, gs, tb, 2, -1, c->stream);
            if (r == cudaSuccess)
                r = launch_fft_axis_fast<float>(reinterpret_cast<cplx<float>*>(nyq), 3, gq, tb, 2, -1, c->stream);
            if (r == cudaSuccess)
                r = launch_divergence_half(reinterpret_cast<const float2*>(spec), nyq, g,
                                           static_cast<const float*>(c->slot_k.p), (float)(-0.5 * kTwoPi / g.dx), tb,
                                           partial, kDiagBlocks, c->stream, &c->launches);
            if (r != cudaSuccess) return r;
            return launch_reduce_final(partial, kDiagBlocks, 2, 0, res + 2 + 2 * half, c->stream, &c->launches);
        });
        if (e != cudaSuccess) return cuda_fail(c, e, "divergence launch");
    }
    CK(c, cudaMemcpyAsync(host, res, 6 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    CK(c, cudaStreamSynchronize(c->stream));
    return PSATD_OK;
}

}  // namespace

psatd_status psatd_diagnostics(psatd_ctx* c, psatd_diag* out) {
    psatd_status st = check_ctx(c, true, true);
    if (st) return st;
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "not allowed while a batch is being captured");
    if (!out) return fail(c, PSATD_ERR_ARG, "NULL out");
    if (c->real_fields) {
        double host[6];
        st = diagnostics_real(c, host);
        if (st) return st;
        out->energy_E = host[0];
        out->energy_B = host[1];
        out->energy = host[0] + host[1];
        out->max_div_E = host[2];
        out->max_E_hat = host[3];
        out->max_div_B = host[4];
        out->max_B_hat = host[5];
        return check_device_error(c);
    }
    const size_t n = n_cells(c->grid);
    const size_t es = cplx_size(c->prec);
    CK(c, ensure_buf(c->diag_spec, 3 * n * es));
    CK(c, ensure_buf(c->diag_partial, (size_t)kDiagBlocks * 2 * sizeof(double)));
    CK(c, ensure_buf(c->diag_out, 8 * sizeof(double)));
    double* partial = static_cast<double*>(c->diag_partial.p);
    double* res = static_cast<double*>(c->diag_out.p);
    double host[6];
    const GridGeom g = geom(c);
    cudaError_t e = timed(c, PSATD_KERNEL_DIAG, [&] {
        cudaError_t r = c->prec == 64
            ? launch_energy<double>(static_cast<const cplx<double>*>(c->fields), n, partial, kDiagBlocks, c->stream, &c->launches)
            : launch_energy<float>(static_cast<const cplx<float>*>(c->fields), n, partial, kDiagBlocks, c->stream, &c->launches);
        if (r != cudaSuccess) return r;
        return launch_reduce_final(partial, kDiagBlocks, 2, 2, res, c->stream, &c->launches);
    });
    if (e != cudaSuccess) return cuda_fail(c, e, "energy launch");
    for (int half = 0; half < 2; ++half) {
        const char* src = static_cast<const char*>(c->fields) + (size_t)3 * half * n * es;
        CK(c, cudaMemcpyAsync(c->diag_spec.p, src, 3 * n * es, cudaMemcpyDeviceToDevice, c->stream));
        if (c->prec == 64) e = fft3d<double>(c, static_cast<cplx<double>*>(c->diag_spec.p), 3, -1, PSATD_KERNEL_DIAG);
        else e = fft3d<float>(c, static_cast<cplx<float>*>(c->diag_spec.p), 3, -1, PSATD_KERNEL_DIAG);
        if (e != cudaSuccess) return cuda_fail(c, e, "divergence fft launch");
        e = timed(c, PSATD_KERNEL_DIAG, [&] {
            cudaError_t r = c->prec == 64
                ? launch_divergence<double>(static_cast<const cplx<double>*>(c->diag_spec.p), g, tables<double>(c), partial, kDiagBlocks, c->stream, &c->launches)
                : launch_divergence<float>(static_cast<const cplx<float>*>(c->diag_spec.p), g, tables<float>(c), partial, kDiagBlocks, c->stream, &c->launches);
            if (r != cudaSuccess) return r;
            return launch_reduce_final(partial, kDiagBlocks, 2, 0, res + 2 + 2 * half, c->stream, &c->launches);
        });
        if (e != cudaSuccess) return cuda_fail(c, e, "divergence launch");
    }
    CK(c, cudaMemcpyAsync(host, res, 6 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    CK(c, cudaStreamSynchronize(c->stream));
    out->energy_E = host[0];
    out->energy_B = host[1];
    out->energy = host[0] + host[1];
    out->max_div_E = host[2];
    out->max_E_hat = host[3];
    out->max_div_B = host[4];
    out->max_B_hat = host[5];
    return check_device_error(c);
}

double psatd_time(const psatd_ctx* c) { return c ? c->t : 0.0; }

psatd_status psatd_set_time(psatd_ctx* c, double t) {
    if (!c) return fail(nullptr, PSATD_ERR_ARG, "NULL context");
    if (!is_finite(t)) return fail(c, PSATD_ERR_ARG, "t must be finite");
    c->t = t;
    return PSATD_OK;
}

psatd_status psatd_synchronize(psatd_ctx* c) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "cannot synchronise while a batch is being captured");
    CK(c, cudaStreamSynchronize(c->stream));
    return check_device_error(c);
}

long long psatd_launch_count(const psatd_ctx* c) { return c ? c->launches : 0; }

psatd_status psatd_selftest_wait_timeout(psatd_ctx* c) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    CK(c, launch_wait_timeout_selftest(c->dev_err, c->stream));
    ++c->launches;
    return psatd_synchronize(c);
}

psatd_status psatd_batch_begin(void* cuda_stream, psatd_batch** out) {
    if (!out) return fail(nullptr, PSATD_ERR_ARG, "NULL out");
    *out = nullptr;
    if (g_capture) return fail(nullptr, PSATD_ERR_STATE, "a batch is already being captured on this thread");
    psatd_batch* b = new (std::nothrow) psatd_batch();
    if (!b) return fail(nullptr, PSATD_ERR_OOM, "host allocation failed");
    b->stream = static_cast<cudaStream_t>(cuda_stream);
    if (!b->stream) {
        delete b;
        return fail(nullptr, PSATD_ERR_ARG, "a batch needs a non-default stream");
    }
    cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        delete b;
        return cuda_fail(nullptr, e, "cudaStreamBeginCapture");
    }
    b->capturing = true;
    g_capture = b;
    *out = b;
    return PSATD_OK;
}

psatd_status psatd_batch_end(psatd_batch* b) {
    if (!b || !b->capturing) return fail(nullptr, PSATD_ERR_ARG, "batch is not capturing");
    b->capturing = false;
    g_capture = nullptr;
    cudaError_t e = cudaStreamEndCapture(b->stream, &b->graph);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&b->exec, b->graph, 0);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGraphInstantiate");
    return PSATD_OK;
}

psatd_status psatd_batch_launch(psatd_batch* b) {
    if (!b || !b->exec) return fail(nullptr, PSATD_ERR_STATE, "batch has no instantiated graph");
    cudaError_t e = cudaGraphLaunch(b->exec, b->stream);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGraphLaunch");
    for (auto& p : b->time_advance) p.first->t += p.second;
    for (auto& p : b->time_set) p.first->t = p.second;
    return PSATD_OK;
}

long long psatd_batch_nodes(const psatd_batch* b) {
    if (!b || !b->graph) return 0;
    size_t n = 0;
    if (cudaGraphGetNodes(b->graph, nullptr, &n) != cudaSuccess) return 0;
    return (long long)n;
}

void psatd_batch_destroy(psatd_batch* b) {
    if (!b) return;
    if (b->capturing) {
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(b->stream, &g);
        if (g) cudaGraphDestroy(g);
        if (g_capture == b) g_capture = nullptr;
    }
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    delete b;
}

psatd_status psatd_autotune(psatd_ctx* c, int trial_steps, int* path_out, int* shift_out, double* ms_out) {
    psatd_status st = check_ctx(c, true, true);
    if (st) return st;
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "cannot tune inside a batch capture");
    if (c->real_fields) {                      // one kernel set: nothing to choose
        if (path_out) *path_out = PSATD_PATH_AUTO;
        if (shift_out) *shift_out = 0;
        if (ms_out) *ms_out = -1.0;
        return PSATD_OK;
    }
    if (trial_steps < 1) trial_steps = 2;
    const auto key = std::make_tuple(c->grid.Nx, c->grid.Ny, c->grid.Nz, c->prec);
    {
        std::lock_guard<std::mutex> lock(g_tuned_mutex);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end()) {
            c->kernel_path = it->second.first;
            c->tile_shift = it->second.second;
            if (path_out) *path_out = c->kernel_path;
            if (shift_out) *shift_out = c->tile_shift;
            if (ms_out) *ms_out = -1.0;
            return PSATD_OK;
        }
    }
    // trial runs on a scratch copy so the context's fields stay untouched
    void* scratch = nullptr;
    CK(c, lib_malloc(&scratch, c->field_bytes));
    void* saved = c->fields;
    const double t_saved = c->t;
    const bool prof_saved = c->prof_on;
    c->prof_on = false;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int best_path = c->kernel_path, best_shift = c->tile_shift;
    double best_ms = 1e300;
    cudaError_t err = cudaMemcpyAsync(scratch, saved, c->field_bytes, cudaMemcpyDeviceToDevice, c->stream);
    c->fields = scratch;
    const int paths[3] = {PSATD_PATH_AUTO, PSATD_PATH_REGISTER, PSATD_PATH_GENERIC};
    for (int pi = 0; pi < 3 && err == cudaSuccess; ++pi) {
        for (int sh = -1; sh <= 1 && err == cudaSuccess; ++sh) {
            c->kernel_path = paths[pi];
            c->tile_shift = sh;
            for (int w = 0; w < 1 && err == cudaSuccess; ++w)
                err = c->prec == 64 ? spectral_pass<double>(c, KS_ROTATE, 0.0) : spectral_pass<float>(c, KS_ROTATE, 0.0);
            if (err == cudaSuccess) err = cudaEventRecord(e0, c->stream);
            for (int k = 0; k < trial_steps && err == cudaSuccess; ++k)
                err = c->prec == 64 ? spectral_pass<double>(c, KS_ROTATE, 0.0) : spectral_pass<float>(c, KS_ROTATE, 0.0);
            if (err == cudaSuccess) err = cudaEventRecord(e1, c->stream);
            if (err == cudaSuccess) err = cudaEventSynchronize(e1);
            float ms = 0.f;
            if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
            if (err == cudaSuccess && ms / trial_steps < best_ms) {
                best_ms = ms / trial_steps;
                best_path = paths[pi];
                best_shift = sh;
            }
        }
    }
    c->fields = saved;
    c->field_map_ptr = nullptr;        // the tensor map was last encoded for the scratch copy
    c->t = t_saved;
    c->prof_on = prof_saved;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamSynchronize(c->stream);
    lib_free(scratch);
    if (err != cudaSuccess) return cuda_fail(c, err, "autotune trial");
    c->kernel_path = best_path;
    c->tile_shift = best_shift;
    {
        std::lock_guard<std::mutex> lock(g_tuned_mutex);
        g_tuned[key] = {best_path, best_shift};
    }
    if (path_out) *path_out = best_path;
    if (shift_out) *shift_out = best_shift;
    if (ms_out) *ms_out = best_ms;
    return PSATD_OK;
}

psatd_status psatd_set_kernel_path(psatd_ctx* c, int path) {
    if (!c) return fail(nullptr, PSATD_ERR_ARG, "NULL context");
    if (path != PSATD_PATH_AUTO && path != PSATD_PATH_GENERIC && path != PSATD_PATH_REGISTER)
        return fail(c, PSATD_ERR_ARG, "unknown kernel path");
    c->kernel_path = path;
    return PSATD_OK;
}

psatd_status psatd_profile_enable(psatd_ctx* c, int enable) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    CK(c, harvest(c, c->pending.size()));
    for (int k = 0; k < PSATD_KERNEL_KINDS; ++k) { c->prof_ms[k] = 0.0; c->prof_n[k] = 0; }
    c->prof_on = enable != 0;
    return PSATD_OK;
}

psatd_status psatd_profile_read(psatd_ctx* c, int kind, double* total_ms, long long* launches) {
    psatd_status st = check_ctx(c, false);
    if (st) return st;
    if (kind < 0 || kind >= PSATD_KERNEL_KINDS) return fail(c, PSATD_ERR_ARG, "unknown kernel kind");
    CK(c, harvest(c, c->pending.size()));
    if (total_ms) *total_ms = c->prof_ms[kind];
    if (launches) *launches = c->prof_n[kind];
    return PSATD_OK;
}

const char* psatd_kernel_name(int kind) {
    static const char* names[PSATD_KERNEL_KINDS] = {"fft_x", "fft_y", "fft_z", "kspace_z",
                                                    "init_pulse", "sample_plane", "diagnostics",
                                                    "plane_xy"};
    return (kind >= 0 && kind < PSATD_KERNEL_KINDS) ? names[kind] : "unknown";
}

psatd_status psatd_multi_advance(psatd_ctx* const* ctxs, int n_ctx, const int* n_steps) {
    psatd_status st = multi_check(ctxs, n_ctx);
    if (st) return st;
    psatd_ctx* c0 = ctxs[0];
    if (!n_steps) return fail(c0, PSATD_ERR_ARG, "NULL step counts");
    int nmax = 0;
    for (int p = 0; p < n_ctx; ++p) {
        if (n_steps[p] < 0) return fail(c0, PSATD_ERR_ARG, "step counts must be >= 0");
        nmax = std::max(nmax, n_steps[p]);
    }
    if (nmax == 0) return PSATD_OK;
    MultiPrepared m;
    if (c0->prec == 64) {
        if ((st = multi_prepare<double>(ctxs, n_ctx, n_steps, nullptr, nullptr, &m))) return st;
        if ((st = multi_launch<double>(ctxs, n_ctx, nmax, m, kMultiWaitNs, 0))) return st;
    } else {
        if ((st = multi_prepare<float>(ctxs, n_ctx, n_steps, nullptr, nullptr, &m))) return st;
        if ((st = multi_launch<float>(ctxs, n_ctx, nmax, m, kMultiWaitNs, 0))) return st;
    }
    psatd_batch* b = capturing(c0);
    for (int p = 0; p < n_ctx; ++p) {
        if (b) b->time_advance.push_back({ctxs[p], n_steps[p] * ctxs[p]->dt});
        else ctxs[p]->t += n_steps[p] * ctxs[p]->dt;
    }
    return PSATD_OK;
}

psatd_status psatd_multi_autotune(psatd_ctx* const* ctxs, int n_ctx, int trial_steps, double* ms_per_step) {
    psatd_status st = multi_check(ctxs, n_ctx);
    if (st) return st;
    psatd_ctx* c0 = ctxs[0];
    if (trial_steps < 1) return fail(c0, PSATD_ERR_ARG, "trial_steps must be >= 1");
    if (capturing(c0)) return fail(c0, PSATD_ERR_STATE, "cannot tune inside a batch capture");
    // trials run on copies of the fields
    std::vector<size_t> off((size_t)n_ctx + 1, 0);
    for (int p = 0; p < n_ctx; ++p) off[p + 1] = off[p] + (6 * n_cells(ctxs[p]->grid) * cplx_size(c0->prec) + 255) / 256 * 256;
    DevBuf tmp;
    CK(c0, ensure_buf(tmp, off[n_ctx]));
    std::vector<void*> fields((size_t)n_ctx);
    cudaError_t e = cudaSuccess;
    for (int p = 0; p < n_ctx && e == cudaSuccess; ++p) {
        fields[p] = static_cast<char*>(tmp.p) + off[p];
        e = cudaMemcpyAsync(fields[p], ctxs[p]->fields, 6 * n_cells(ctxs[p]->grid) * cplx_size(c0->prec),
                            cudaMemcpyDeviceToDevice, c0->stream);
    }
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (e == cudaSuccess) e = cudaEventCreate(&ev[0]);
    if (e == cudaSuccess) e = cudaEventCreate(&ev[1]);
    const std::vector<int> steps((size_t)n_ctx, trial_steps);
    std::map<int, MultiChoice> cur;
    for (int p = 0; p < n_ctx; ++p)
        for (int a = 0; a < 3; ++a) {
            const int N = axis_n(ctxs[p]->grid, a);
            cur[N] = multi_choice(c0->prec, N);
        }
    double best_ms = -1.0;
    auto trial = [&](double* ms) -> psatd_status {
        MultiPrepared m;
        psatd_status s2 = c0->prec == 64 ? multi_prepare<double>(ctxs, n_ctx, steps.data(), fields.data(), &cur, &m)
                                         : multi_prepare<float>(ctxs, n_ctx, steps.data(), fields.data(), &cur, &m);
        if (s2) return s2;
        CK(c0, cudaEventRecord(ev[0], c0->stream));
        s2 = c0->prec == 64 ? multi_launch<double>(ctxs, n_ctx, trial_steps, m, kMultiWaitNs, 0)
                            : multi_launch<float>(ctxs, n_ctx, trial_steps, m, kMultiWaitNs, 0);
        if (s2) return s2;
        CK(c0, cudaEventRecord(ev[1], c0->stream));
        CK(c0, cudaEventSynchronize(ev[1]));
        float f = 0.f;
        CK(c0, cudaEventElapsedTime(&f, ev[0], ev[1]));
        *ms = f;
        return check_device_error(c0);
    };
    if (e == cudaSuccess) {
        st = trial(&best_ms);                                  // warm-up (first launch of the kernel)
        if (st == PSATD_OK) st = trial(&best_ms);
        // coordinate descent over the axis lengths: each length tries every
        // distinct radix schedule and tile-width scale with the others fixed
        for (auto it = cur.begin(); st == PSATD_OK && it != cur.end(); ++it) {
            const int N = it->first;
            std::vector<AxisPlan> tried;
            MultiChoice best = it->second;
            for (int v = 0; v < kPlanVariants && st == PSATD_OK; ++v) {
                AxisPlan pl;
                if (!make_plan_variant(N, v, &pl)) continue;
                bool dup = false;
                for (const AxisPlan& q : tried) dup = dup || same_plan(q, pl);
                if (dup) continue;
                tried.push_back(pl);
                for (int sc = -1; sc <= 1 && st == PSATD_OK; ++sc) {
                    const MultiChoice ch{v, sc};
                    if (ch == best) continue;
                    it->second = ch;
                    double ms = 0.0;
                    st = trial(&ms);
                    if (st == PSATD_OK && ms < best_ms) {
                        best_ms = ms;
                        best = ch;
                    }
                }
            }
            it->second = best;
        }
    }
    if (ev[0]) cudaEventDestroy(ev[0]);
    if (ev[1]) cudaEventDestroy(ev[1]);
    cudaStreamSynchronize(c0->stream);
    free_buf(tmp);
    c0->multi_sig.clear();                                     // the uploaded boxes point at the freed copies
    if (e != cudaSuccess) return cuda_fail(c0, e, "autotune set-up");
    if (st) return st;
    {
        std::lock_guard<std::mutex> lock(g_multi_mutex);
        for (auto& kv : cur) g_multi_tuned[{c0->prec, kv.first}] = kv.second;
    }
    if (ms_per_step) *ms_per_step = best_ms / trial_steps;
    return PSATD_OK;
}

psatd_status psatd_selftest_grid_barrier_timeout(psatd_ctx* c) {
    psatd_ctx* ctxs[1] = {c};
    psatd_status st = multi_check(ctxs, 1);
    if (st) return st;
    if (capturing(c)) return fail(c, PSATD_ERR_STATE, "not allowed while a batch is being captured");
    MultiPrepared m;
    const int one = 1;
    st = c->prec == 64 ? multi_prepare<double>(ctxs, 1, &one, nullptr, nullptr, &m)
                       : multi_prepare<float>(ctxs, 1, &one, nullptr, nullptr, &m);
    if (st) return st;
    // one extra arrival that never comes: every block's first barrier wait
    // expires after 2 ms
    st = c->prec == 64 ? multi_launch<double>(ctxs, 1, 1, m, 2000000ull, 1)
                       : multi_launch<float>(ctxs, 1, 1, m, 2000000ull, 1);
    if (st) return st;
    return psatd_synchronize(c);
}

void psatd_debug_set_alloc_limit(long long bytes) {
    std::lock_guard<std::mutex> lock(g_alloc_mutex);
    g_alloc_limit = bytes < 0 ? -1 : bytes;
}

long long psatd_debug_alloc_live(void) {
    std::lock_guard<std::mutex> lock(g_alloc_mutex);
    return g_alloc_live;
}

void psatd_debug_inject_cuda_error(int after_calls, int cuda_error) {
    g_inject_error.store(cuda_error);
    g_inject_after.store(after_calls > 0 ? after_calls : 0);
}

long long psatd_debug_bounds_report(long long* first_index, long long* first_bound) {
#ifdef PSATD_DEBUG
    std::lock_guard<std::mutex> lock(g_dbg_mutex);
    if (cudaDeviceSynchronize() != cudaSuccess) return -1;
    long long total = 0;
    bool first = true;
    for (auto fn : dbg_readers()) {
        long long fi = 0, fb = 0;
        const long long n = fn(&fi, &fb);
        if (n < 0) return -1;
        if (n > 0 && first) {
            if (first_index) *first_index = fi;
            if (first_bound) *first_bound = fb;
            first = false;
        }
        total += n;
    }
    return total;
#else
    (void)first_index;
    (void)first_bound;
    return -2;
#endif
}

}  // extern "C"
