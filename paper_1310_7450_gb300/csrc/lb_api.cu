// lb_api.cu -- the C ABI declared in include/lbnlm.h: handle management, state layout, launch
// sequencing of the fused step, field output, residual reduction, checkpointing.
//
// Device layout of a handle (all channels in one allocation per field):
//   every channel c owns planes of P[c] elements (P[c] >= nx*ny[c], padded to 64 elements);
//   base[c] = sum_{c'<c} P[c'] is the channel's plane offset, so a field with k planes keeps
//   plane j of channel c at  k*base[c] + j*P[c].  Populations: 9 planes (ping-pong A/B);
//   delta rho: 1 plane; carried stress (mode 1): 3 planes; stress output: 4 planes; saved
//   velocity: 2 planes.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <new>
#include <type_traits>
#include <vector>

#include "lb_march_plan.h"
#include "lb_step_march.cuh"
#include "lb_step_resident.cuh"
#include "lb_step_tile.cuh"
#include "lb_sweep.cuh"
#include "lb_sweep_pair.cuh"
#include "lb_sweep_smem.cuh"
#include "lbnlm.h"

namespace lbk {
// learned warm start (lb_warmstart.cu)
struct WsChan {
    double G, tau0, theta, gamma_c;
};
cudaError_t launch_ws_closed_form(int n_ch, const WsChan* prm, const double* gx, const int* nys, const int* row_off,
                                  double* rows, double* grid, double* scale, cudaStream_t s);
template <typename T, typename C>
cudaError_t launch_ws_start(int n_ch, int max_ny, int n_sm, const float* pred, const float* t_mu, const float* t_sd,
                            const double* grid, const double* scale, const double* rows, const double* gx, const int* nys,
                            const int* row_off, const long long* base, const long long* P, int nx, int gpbc, T* pop, C* drho,
                            C* sig3, cudaStream_t s);
template <typename F>
cudaError_t launch_ws_targets(int n_ch, const F* fu, const F* fs, const double* grid, const double* scale, const int* nys,
                              const long long* node_off, int nx, float* targets, cudaStream_t s);
extern template cudaError_t launch_step_tile<double, double, 0>(const StepArgs<double, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<double, double, 1>(const StepArgs<double, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, float, 0>(const StepArgs<float, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, float, 1>(const StepArgs<float, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<__nv_bfloat16, float, 0>(const StepArgs<__nv_bfloat16, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<__nv_bfloat16, float, 1>(const StepArgs<__nv_bfloat16, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<double, float, 0>(const StepArgs<double, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<double, float, 1>(const StepArgs<double, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, double, 0>(const StepArgs<float, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, double, 1>(const StepArgs<float, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<double, double, 0, 3>(const StepArgs<double, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<double, double, 1, 3>(const StepArgs<double, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, float, 0, 3>(const StepArgs<float, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, float, 1, 3>(const StepArgs<float, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<__nv_bfloat16, float, 0, 3>(const StepArgs<__nv_bfloat16, float>&, int, size_t,
                                                                         cudaStream_t);
extern template cudaError_t launch_step_tile<__nv_bfloat16, float, 1, 3>(const StepArgs<__nv_bfloat16, float>&, int, size_t,
                                                                         cudaStream_t);
extern template cudaError_t launch_step_tile<double, double, 0, 1>(const StepArgs<double, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<double, double, 0, 2>(const StepArgs<double, double>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, float, 0, 1>(const StepArgs<float, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<float, float, 0, 2>(const StepArgs<float, float>&, int, size_t, cudaStream_t);
extern template cudaError_t launch_step_tile<__nv_bfloat16, float, 0, 1>(const StepArgs<__nv_bfloat16, float>&, int, size_t,
                                                                         cudaStream_t);
extern template cudaError_t launch_step_tile<__nv_bfloat16, float, 0, 2>(const StepArgs<__nv_bfloat16, float>&, int, size_t,
                                                                         cudaStream_t);
#define LB_SWEEP_EXTERN(T, C, NX)                                                                                   \
    extern template cudaError_t launch_sweep<T, C, 128, 4, NX>(const SweepArgs<T, C>&, int, int, size_t, cudaStream_t); \
    extern template cudaError_t launch_sweep<T, C, 256, 4, NX>(const SweepArgs<T, C>&, int, int, size_t, cudaStream_t); \
    extern template cudaError_t launch_sweep_capacity<T, C, 128, 4, NX>(int, size_t, int*);                            \
    extern template cudaError_t launch_sweep_capacity<T, C, 256, 4, NX>(int, size_t, int*);
LB_SWEEP_EXTERN(float, float, 0)
LB_SWEEP_EXTERN(__nv_bfloat16, float, 0)
LB_SWEEP_EXTERN(double, double, 0)
LB_SWEEP_EXTERN(float, float, 4)
LB_SWEEP_EXTERN(__nv_bfloat16, float, 4)
LB_SWEEP_EXTERN(double, double, 4)
#undef LB_SWEEP_EXTERN
#define LB_SWEEP_SMEM_EXTERN(T, C, NX)                                                                                   \
    extern template cudaError_t launch_sweep_smem<T, C, 128, 4, NX>(const SweepArgs<T, C>&, int, int, size_t, cudaStream_t); \
    extern template cudaError_t launch_sweep_smem<T, C, 256, 4, NX>(const SweepArgs<T, C>&, int, int, size_t, cudaStream_t); \
    extern template cudaError_t launch_sweep_smem_capacity<T, C, 128, 4, NX>(int, size_t, int*);                            \
    extern template cudaError_t launch_sweep_smem_capacity<T, C, 256, 4, NX>(int, size_t, int*);
LB_SWEEP_SMEM_EXTERN(double, double, 0)
LB_SWEEP_SMEM_EXTERN(double, double, 4)
#undef LB_SWEEP_SMEM_EXTERN
#define X(T, NT, NX) LB_SWEEP_PAIR(extern, T, NT, NX)
LB_SWEEP_PAIR_VARIANTS(X)
#undef X
#define X(T, SMODE, BND, SCHEME)                                                                              \
    LB_MARCH_STEP(extern, T, SMODE, BND, SCHEME, kFull) LB_MARCH_FIELDS(extern, T, SMODE, BND, SCHEME, kFull) \
    LB_MARCH_STEP(extern, T, SMODE, BND, SCHEME, kPart) LB_MARCH_FIELDS(extern, T, SMODE, BND, SCHEME, kPart) \
    LB_MARCH_STEP(extern, T, SMODE, BND, SCHEME, kOdd) LB_MARCH_FIELDS(extern, T, SMODE, BND, SCHEME, kOdd)
LB_MARCH_VARIANTS(X, float)
LB_MARCH_VARIANTS(X, __nv_bfloat16)
#undef X
#define X(T, C, SMODE, NT) LB_RESIDENT(extern, T, C, SMODE, NT)
LB_RESIDENT_VARIANTS(X)
#undef X
}  // namespace lbk

using namespace lbk;

namespace {

thread_local char g_err[512] = "";

lb_status fail(lb_status s, const char* fmt, const char* detail = nullptr) {
    std::snprintf(g_err, sizeof g_err, fmt, detail ? detail : "");
    return s;
}
}  // namespace

namespace lbk {
// Lets other translation units of the library report a failure through lb_last_error().
void set_last_error(const char* msg) { std::snprintf(g_err, sizeof g_err, "%s", msg); }
}  // namespace lbk

namespace {

lb_status cuda_fail(cudaError_t e, const char* where) {
    std::snprintf(g_err, sizeof g_err, "%s: %s", where, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA;
}
#define LB_CK(call)                                              \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);      \
    } while (0)

constexpr int kThreads = 256;        // threads per CTA of the tile kernel
constexpr double kGuard = 0.3;       // |u| above which a channel is declared unstable

// SplitMix64 (Steele, Lea & Flood 2014; 64-bit finaliser as published by Vigna): output number
// `counter` (>= 1) of the stream seeded with `seed`.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t counter) {
    uint64_t z = seed + counter * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

struct InitChan {
    long long base, P;
    int ny, gpbc;
    double rho0, amp;
    uint64_t seed;
    double rho_in, rho_out;  // GPBC: densities at the ghost columns x = -1 and x = nx
};

// Rest equilibrium n_i = w_i rho(r), rho = rho0 (1 + amp U(-1,1)); delta rho = 0.  Under GPBC the
// density starts on the straight line between the inlet and outlet ghost densities (the linear
// pre-initialisation of Sec. II B): rho = rho_in + (rho_out - rho_in)(x+1)/(nx+1) + rho0 amp U.
template <typename T, typename C>
__global__ void k_init(T* pop, C* drho, C* sig3, const InitChan* ch, int nx, int smode) {
    const InitChan c = ch[blockIdx.y];
    const long long n = (long long)nx * c.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double rho = c.rho0;
        double U = 0.0;
        if (c.amp != 0.0) {
            const uint64_t z = splitmix64(c.seed, (uint64_t)k + 1ull);
            U = __dadd_rn(__dmul_rn((double)(z >> 11), 0x1p-52), -1.0);
            rho = __dmul_rn(c.rho0, __dadd_rn(1.0, __dmul_rn(c.amp, U)));
        }
        if (c.gpbc) {
            const double lin = c.rho_in + (c.rho_out - c.rho_in) * (double)(k % nx + 1) / (double)(nx + 1);
            rho = __dadd_rn(lin, __dmul_rn(c.rho0, __dmul_rn(c.amp, U)));
        }
        const double dev = rho - 1.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) Store<T>::st(pop + 9 * c.base + i * c.P + k, (C)(wgt<double>(i) * dev));
        drho[c.base + k] = C(0);
        if (smode == 1)
            for (int j = 0; j < 3; ++j) sig3[3 * c.base + j * c.P + k] = C(0);
    }
}

// Populations <-> full FP64 values in plane order (host staging is compact per channel).
template <typename T, typename C>
__global__ void k_pop_from_f64(T* pop, const double* src, const long long* base, const long long* P,
                               const long long* node_off, const int* ny, int nx) {
    const int c = blockIdx.y;
    const long long n = (long long)nx * ny[c];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
#pragma unroll
        for (int i = 0; i < 9; ++i)
            Store<T>::st(pop + 9 * base[c] + i * P[c] + k, (C)(src[9 * node_off[c] + i * n + k] - wgt<double>(i)));
}
template <typename T, typename C>
__global__ void k_pop_to_f64(const T* pop, double* dst, const long long* base, const long long* P,
                             const long long* node_off, const int* ny, int nx) {
    const int c = blockIdx.y;
    const long long n = (long long)nx * ny[c];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
#pragma unroll
        for (int i = 0; i < 9; ++i)
            dst[9 * node_off[c] + i * n + k] = (double)Store<T>::ld(pop + 9 * base[c] + i * P[c] + k) + wgt<double>(i);
}
// k planes of a compact per-channel FP64 field <-> the padded C planes.
template <typename C>
__global__ void k_planes_from_f64(C* dst, const double* src, int kp, const long long* base, const long long* P,
                                  const long long* node_off, const int* ny, int nx) {
    const int c = blockIdx.y;
    const long long n = (long long)nx * ny[c];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        for (int j = 0; j < kp; ++j) dst[kp * base[c] + j * P[c] + k] = (C)src[kp * node_off[c] + j * n + k];
}
template <typename C>
__global__ void k_planes_to_f64(const C* src, double* dst, int kp, const long long* base, const long long* P,
                                const long long* node_off, const int* ny, int nx) {
    const int c = blockIdx.y;
    const long long n = (long long)nx * ny[c];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        for (int j = 0; j < kp; ++j) dst[kp * node_off[c] + j * n + k] = (double)src[kp * base[c] + j * P[c] + k];
}

// Warm start: equilibrium of (rho, u - f/(2 rho)) so that j = sum c n + f/2 = rho u (Eq. rhoj).
template <typename T, typename C>
__global__ void k_set_fields(T* pop, C* drho, C* sig3, const double* u, const double* rho, const double* dr,
                             const long long* base, const long long* P, const long long* node_off, const int* ny,
                             const double* gx, int nx, int smode, int gpbc) {
    const int c = blockIdx.y;
    const double g = gpbc ? 0.0 : gx[c];  // no body force in a pressure-driven channel
    const long long n = (long long)nx * ny[c];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const long long node = node_off[c] + k;
        const double r = rho[node];
        const double ux = u[2 * node] - 0.5 * g / r, uy = u[2 * node + 1];
        const double usq = ux * ux + uy * uy;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double cu = cx(i) * ux + cy(i) * uy;
            const double w = wgt<double>(i);
            const double dev = w * ((r - 1.0) + r * (3.0 * cu + 4.5 * cu * cu - 1.5 * usq));
            Store<T>::st(pop + 9 * base[c] + i * P[c] + k, (C)dev);
        }
        drho[base[c] + k] = (dr && !gpbc) ? (C)dr[node] : C(0);
        if (smode == 1)
            for (int j = 0; j < 3; ++j) sig3[3 * base[c] + j * P[c] + k] = C(0);
    }
}

// Give channels c0 .. c0 + n - 1 the body force (or, WALL, the moving wall's velocity) v, and keep a
// device copy in gx for the kernels that read the drive there.  A call sets one channel or all of them, to
// one value: an argument, so nothing is read from host memory and no staging has to be kept until the
// kernel ran; launched while the kernel before it still runs (what it reads before the wait is constant
// after create).  Sixteen steps of 1024 x 1024 FP32 whose drive changes and whose monitor is copied to
// device memory every step, and the fields: 531 us with a mapped staging slot, an event and a copy, 452
// now.  A force for all of 20 000 channels: 354 us in launches of 128 channels' values, 26 now.
constexpr int kDriveThreads = 128;
template <typename C, bool WALL>
__global__ void __launch_bounds__(kDriveThreads) k_apply_drive(ChanParams<C>* chan, double* gx, double v, int c0, int n, int n_ch,
                                                               int nx) {
    const int k = blockIdx.x * kDriveThreads + threadIdx.x, c = c0 + k;
    const bool on = k < n, gpbc = !WALL && on && chan[c].gpbc;
    const C rho0 = gpbc ? chan[c].rho0_m1 : C(0);
    grid_dependency();
    if (!on) return;
    if (WALL) {
        gx[n_ch + c] = v;
        chan[c].u_wall = (C)v;
        return;
    }
    gx[c] = v;
    if (gpbc) {  // pressure-driven: v sets the ghost densities, there is no body force
        const double half = 1.5 * v * (double)(nx + 1);
        chan[c].rho_in = (C)((double)rho0 + half);
        chan[c].rho_out = (C)((double)rho0 - half);
    } else {
        chan[c].gx = (C)v;
    }
}

// Copy n doubles of device memory to mapped pinned host memory or to device memory (the monitor's
// way out: no copy-engine transfer in the stream, and set up while the step before it runs).  20 000
// channels (640 KB) to device memory: 102 us by one block of 128 threads, 2.8 by one thread per value.
__global__ void k_copy_out(const double* src, double* dst, int n) {
    grid_dependency();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) dst[k] = src[k];
}
cudaError_t copy_out(const double* src, double* dst, int n, cudaStream_t s) {
    return launch_dependent(true, k_copy_out, (n + 127) / 128, 128, 0, s, src, dst, n);
}

// Per-channel reduction of the step's block partials, one warp per channel in a fixed order
// (deterministic; the row-march kernel forms the same values itself, see monitor_reduce).
// with_residual = 0: the partials hold flux and max |u| only (F_MON); the residual slot reads -1
__global__ void k_reduce_residual(const double* partials, const int* item_begin, const int* status, double* mon,
                                  int nx, long long state_index, int with_residual) {
    const int c = blockIdx.x;
    monitor_reduce(partials, item_begin[c], item_begin[c + 1], status[c], mon + 4 * c, nx, state_index, with_residual,
                   threadIdx.x, false);
}

int grid_for(long long n) {
    long long b = (n + 255) / 256;
    return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

// Storage type T and arithmetic type C of a precision mode.
template <typename X> struct Tag { using type = X; };
template <typename F>
auto with_types(int prec, F&& f) {
    switch (prec) {
        case LB_PREC_F64: return f(Tag<double>{}, Tag<double>{});
        case LB_PREC_F32: return f(Tag<float>{}, Tag<float>{});
        case LB_PREC_BF16: return f(Tag<__nv_bfloat16>{}, Tag<float>{});
        case LB_PREC_F64S_F32M: return f(Tag<double>{}, Tag<float>{});
        default: return f(Tag<float>{}, Tag<double>{});
    }
}
#define LB_TYPES(tt, tc)                          \
    using T = typename decltype(tt)::type;        \
    using C = typename decltype(tc)::type;

}  // namespace

// Channels of one width class in the batched sweep and the configuration they run with.
struct SweepGroup {
    int cls = 0;                    // floor(log2 ny)
    int begin = 0, count = 0;       // range in the widest-first channel order
    int ny_min = 0, ny_max = 0;
    int var = 0, nt = 0, cl = 0;    // 0: state through L2, 1: state in shared memory; nt == 0: not tuned
    double tune_ms = 0.0;
};

// NVTX range over a public call, so that profiler timelines (Nsight Systems / Compute) group the
// launches of one lb_step or sweep; a no-op unless a tool is attached.
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

constexpr unsigned long long kDefaultWaitNs = 2000000000ull;
constexpr long kResidentSteps = 6;

struct lb_handle {
    int dev = 0;
    cudaStream_t stream = nullptr;
    int n_ch = 0, nx = 0, prec = 0, smode = 0, flags = 0;
    std::vector<int> ny;
    std::vector<long long> P, base, node_off;
    long long planes = 0;  // sum of P
    long long nodes = 0;
    std::vector<lb_params> params;
    size_t tsize = 0, csize = 0;  // storage / arithmetic element sizes
    // device state
    void *popA = nullptr, *popB = nullptr, *drho = nullptr, *sig3 = nullptr, *sig4 = nullptr, *uprev = nullptr;
    void* snn = nullptr;  // stress-divergence scheme: Sigma^nN of the current step [3 planes]
    void* phi = nullptr;  // relaxation-time extensions: fluidity 1/tau_M per node [plane]
    int scheme = 0;       // 0: the paper's forcing; 1: generalized Newtonian; 2: div Sigma^nN force;
                          // 3: the paper's forcing with the relaxation-time extensions
    std::vector<double> beta_rho, rho_ref, tau_f;  // scheme 3, per channel
    // learned warm start: per-channel closed-form parameters, row offsets, closed form on the rows
    // [row][3] and on the network grid [channel][3][256], scales [channel][3]
    void *ws_prm = nullptr, *ws_row_off = nullptr, *ws_rows = nullptr, *ws_grid = nullptr, *ws_scale = nullptr;
    bool ws_ready = false;     // ... allocated and filled
    void* chan = nullptr;
    WorkItem* items_d = nullptr;
    int* item_begin_d = nullptr;
    double* partials = nullptr;
    double* mon_d = nullptr;
    int* status_d = nullptr;
    long long *base_d = nullptr, *P_d = nullptr, *node_off_d = nullptr;
    int* ny_d = nullptr;
    double* gx_d = nullptr;
    void* fields[2] = {nullptr, nullptr};  // staging of fields as float / double, 7 values per node (each allocated
                                           // when first needed and kept: a captured call holds its address)
    void* hstage = nullptr;    // device staging for FP64 host transfers
    size_t hstage_bytes = 0;
    // launch plan
    std::vector<WorkItem> items;
    std::vector<int> item_begin;
    size_t smem = 0;
    // bookkeeping
    long step = 0;
    long uprev_state = -10;    // state index whose velocity u_prev holds
    long mon_state = -1;       // state index of the last monitor evaluation (-1: none)
    bool mon_resid = false;    // the last monitor evaluation includes the residual
    int monitor_mode = 0;      // LB_MONITOR_RESIDUAL or LB_MONITOR_FLUX_MAX
    int* status_h = nullptr;   // pinned, mapped (row march: the kernel's status mirror)
    int* status_hd = nullptr;  // its device address
    double* mon_h = nullptr;   // mapped pinned copy of the monitor for lb_monitor
    double* mon_hd = nullptr;
    cudaEvent_t status_ev = nullptr;
    bool status_pending = false;
    bool any_unstable = false;
    bool any_timeout = false;
    unsigned long long wait_ns = kDefaultWaitNs;  // limit of the row-march kernel's mbarrier waits
    // row-march kernel (large single channels, FP32 / BF16 storage)
    bool march = false;
    int march_strip = kFull;   // its strips: whole, partial, or rows of any length
    CUtensorMap mapA, mapB;    // tensor maps of the two population buffers ...
    const void* mapA_buf = nullptr;  // ... and the buffers they describe (the pointers swap)
    const void* mapB_buf = nullptr;
    // persistent cluster sweep
    long long* sweep_steps_d = nullptr;
    double* sweep_res_d = nullptr;
    int* sweep_order_d = nullptr;
    std::vector<SweepGroup> sweep_groups;  // width classes of the active channels and their configurations
    std::vector<cudaStream_t> gstreams;     // forked streams of the class launches
    std::vector<cudaEvent_t> gevents;
    cudaEvent_t fork_ev = nullptr;
    bool sweep_fixed = false;               // configuration set by lb_sweep_set_config
    cudaGraphExec_t sweep_gexec = nullptr;  // the class launches captured as one graph ...
    std::vector<double> sweep_key;          // ... for these arguments and configurations
    const void* sweep_pin = nullptr;        // ... and this population buffer
    MarchItem* march_items_d = nullptr;
    int n_march_items = 0, march_grid = 0;
    // resident stepping of a small single channel: CTAs of its cluster (0: not used), threads, shared memory
    int res_cl = 0, res_threads = 0;
    size_t res_smem = 0;
    // CUDA graphs of kGraphSteps plain tile-kernel steps, one per input buffer (an even count of
    // steps leaves the buffers where they were, so each graph starts from the buffer it names)
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};
    const void* gexec_pin[2] = {nullptr, nullptr};
    cudaStream_t cap_stream = nullptr;
    long graph_replays = 0;
    // generalized periodic boundaries (x_mode LB_X_GPBC)
    bool gpbc = false;
    void* gcol = nullptr;  // boundary-column moments and means (see StepArgs::gcol)
    double* gpart = nullptr;    // per-block partial sums of the column kernel
    unsigned* gcount = nullptr; // per-column block counters (zero between launches)
    unsigned* done_count_d = nullptr;  // row-march CTAs done with the launch (zero between launches)
    int gpbc_max_ny = 0;
    int gny = 0;           // sum of ny over the channels
    std::vector<int> row_off;
    // planar Couette flow (walls LB_WALLS_COUETTE): Zou-He moving wall on the last row
    bool moving = false;
    std::vector<double> u_wall;
};

namespace {

template <typename C>
std::vector<ChanParams<C>> make_chan(const lb_handle* h) {
    std::vector<ChanParams<C>> v(h->n_ch);
    for (int c = 0; c < h->n_ch; ++c) {
        const lb_params& p = h->params[c];
        ChanParams<C> q{};
        q.base = h->base[c];
        q.P = h->P[c];
        q.node_off = h->node_off[c];
        q.ny = h->ny[c];
        q.omega = (C)(1.0 / p.tau_lb);
        q.k1 = (C)(-9.0 / (2.0 * p.tau_lb));
        q.k2 = (C)(1.0 - 1.0 / (2.0 * p.tau_lb));
        q.gx = (C)p.g_x;
        q.G = (C)p.G_inf;
        q.tau = (C)(p.theta * p.tau0);
        q.inv_gc = std::isinf(p.gamma_c) ? C(0) : (C)(1.0 / p.gamma_c);
        q.cD = (C)(p.G_inf * p.tau0 - p.rho0 * (p.tau_lb - 0.5) / 3.0);
        q.kdr = C(1);
        q.rho0_m1 = (C)(p.rho0 - 1.0);
        q.moving = h->moving ? 1 : 0;
        q.u_wall = (C)h->u_wall[c];
        q.scheme = h->scheme;
        q.rho_ref = C(1);
        if (h->scheme == 3) {
            q.beta_rho = (C)h->beta_rho[c];
            q.rho_ref = (C)h->rho_ref[c];
            q.tau_f = (C)h->tau_f[c];
        }
        if (h->scheme == 1 || h->scheme == 2) {
            // the comparison schemes of Sec. II C: no stress line and no flow-induced density
            q.k1 = C(0);
            q.kdr = C(0);
            q.gn_a = (C)(3.0 * p.G_inf / p.rho0);
            q.gn_b = (C)(0.5 + 3.0 * p.G_inf * p.tau0 / p.rho0);
        }
        if (h->gpbc) {
            // GPBC (Sec. II B): the pressure gradient replaces the body force, p_+ - p_- = g (nx+1)
            // between the ghost columns; no flow-induced density, Eq. (bodyforce) first line only
            q.gpbc = 1;
            q.row_off = h->row_off[c];
            q.kdr = C(0);
            q.gx = C(0);
            q.rho_in = (C)((p.rho0 - 1.0) + 1.5 * p.g_x * (double)(h->nx + 1));
            q.rho_out = (C)((p.rho0 - 1.0) - 1.5 * p.g_x * (double)(h->nx + 1));
        }
        q.tau_c = std::min(C(0.5) * q.tau * q.inv_gc, std::numeric_limits<C>::max());  // (finite: times no shear it is 0)
        q.cDh = C(0.5) * q.cD;
        q.m15k = C(-1.5) * q.kdr;
        q.om3 = C(3) * q.omega;
        q.om15 = C(-1.5) * q.omega;
        q.om45 = C(4.5) * q.omega;
        q.k23 = C(3) * q.k2;
        q.k245 = C(4.5) * q.k2;
        q.k1h = C(0.5) * q.k1;
        q.k12 = C(2) * q.k1;
        v[c] = q;
    }
    return v;
}

// Tile plan: narrow channels (nx <= 64) use full-width tiles of at most kThreads/nx (>= 4) rows;
// wide ones 32 x 8 tiles.  Row tiles are balanced: with ny >= 3 and a row target >= 4 every tile
// gets between 2 and the target rows (one-sided differences at a wall need the two rows next to
// it inside the tile or its halo), so a tile never holds more nodes than the CTA has threads.
// FP64 arithmetic: a tile's time is its SM's FP64 operations, so the row tiles are made more and shorter until their
// number is the next multiple of the SMs (4 x 64: one tile -> 32; 256 x 257: 264 -> 304, two on every SM
// instead of two on some).
void plan_tiles(lb_handle* h, int n_sm) {
    h->items.clear();
    h->item_begin.assign(h->n_ch + 1, 0);
    int maxEX = 0, maxEY = 0;
    int nxt = 32, nyt_target = kThreads / 32;
    if (h->nx <= kThreads / 4) { nxt = h->nx; nyt_target = kThreads / h->nx; }
    const int ntx = (h->nx + nxt - 1) / nxt;
    long long total = 0;
    for (int ny : h->ny) total += (long long)ntx * ((ny + nyt_target - 1) / nyt_target);
    const double finer = h->csize == 8 ? (double)((total + n_sm - 1) / n_sm * n_sm) / (double)total : 1.0;
    for (int c = 0; c < h->n_ch; ++c) {
        h->item_begin[c] = (int)h->items.size();
        const int ny = h->ny[c];
        const int base = (ny + nyt_target - 1) / nyt_target;
        const int nty = std::max(base, std::min(ny / 2, (int)(base * finer)));
        for (int ty = 0; ty < nty; ++ty) {
            const int y0 = (int)((long long)ny * ty / nty), y1 = (int)((long long)ny * (ty + 1) / nty);
            for (int tx = 0; tx < ntx; ++tx) {
                WorkItem w{};
                w.ch = c;
                w.x0 = tx * nxt;
                w.nxt = (tx == ntx - 1) ? h->nx - w.x0 : nxt;
                if (ntx == 1) w.nxt = h->nx;
                w.y0 = y0;
                w.nyt = y1 - y0;
                h->items.push_back(w);
                const int EX = (w.nxt == h->nx) ? h->nx : w.nxt + 2;
                if (EX > maxEX) maxEX = EX;
                if (w.nyt + 2 > maxEY) maxEY = w.nyt + 2;
            }
        }
    }
    h->item_begin[h->n_ch] = (int)h->items.size();
    h->smem = (size_t)maxEX * maxEY * 2 * h->csize;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)f;
    }
    return fn;
}

// 3-D map over the 9 population planes of channel 0: dims (nx, ny, 9), box (strip, 1, 9); where the row length is
// no multiple of 16 bytes the planes are one row each: dims (nx ny, 1, 9).
bool make_pop_map(const lb_handle* h, void* base, CUtensorMap* map) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const bool bf = h->prec == LB_PREC_BF16, odd = h->march_strip == kOdd;
    const cuuint64_t es = bf ? 2 : 4, plane = (cuuint64_t)h->P[0] * es;
    const int width = bf ? march_slot_width<__nv_bfloat16>(kMarchW, odd) : march_slot_width<float>(kMarchW, odd);
    cuuint64_t dims[3] = {(cuuint64_t)h->nx * (odd ? h->ny[0] : 1), odd ? 1 : (cuuint64_t)h->ny[0], 9};
    cuuint64_t strides[2] = {odd ? plane : (cuuint64_t)h->nx * es, plane};
    cuuint32_t box[3] = {(cuuint32_t)width, 1, 9};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(map, bf ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Programmatic dependent launch takes about 2 us off a march step, but lets blocks land on whichever SM frees a
// slot first, against the plan that deals rows by a block's rank on its SM.  us per step without / with:
// FP32 1024 x 1024 22.5 / 20.7, 2048 x 2048 72.6 / 71.2, 4096 x 4096 252 / 257; BF16 1024 x 1024 20.7 / 20.1,
// 8192 x 2048 214 / 236.  With pressure-driven ends (a column kernel before every step): FP32 2048 x 1000 52.0 / 56.5; BF16 2048 x 1000 47.0 / 43.8, 256 x 8192 63.2 / 60.7, 4096 x 4096 257.6 / 255.7.
static bool march_dependent(int prec, bool gpbc, long long nodes) {
    if (gpbc) return prec == LB_PREC_BF16;
    return nodes <= (prec == LB_PREC_BF16 ? 1 << 21 : 1 << 22);
}

// Constants measured with six CTAs of two warps per SM (us per step, one GPU):
//   FP32 4096 x 4096: skew 0.06: 251.9, 0.12: 252.9, 0: 252.7, 0.2: 257.7; f = 1.2 252.9, 1.05: 264.0,
//     1.35: 253.6; pressure-driven ends at 2048 x 1000 f = 1.7: 51.8, 1.5: 53.7, 1.3: 55.5, 1.2: 59.7.
//   BF16 8192 x 2048: skew 0.3 f = 1.15: 214.4; f = 1.3: 212.8 (but leaves CTAs idle with eight per SM); f = 1.05: 228.4; skew 0.15 / 0.22 with
//     f = 1.15: 214.5 / 214.9; skew 0.4: 228.6.
//   BF16, pressure-driven ends, 4096 x 4096 / 2048 x 1000 / 256 x 8192 / 640 x 4096: skew 0.16 f = 1.4: 251.4 / 45.7 /
//     60.9 / 63.0; f = 1.3: 261.8 / 47.6 / 61.0 / 64.3; f = 1.5: 255.5 / 45.1 / 60.8 / 62.2; skew 0.3, 1.5: 251.1 / 45.7 / 61.9 /
//     63.0; skew 0, 1.4: 262.3 / 45.6 / 61.0 / 62.6.
//   BF16 grids whose steps are launched while the one before runs: blocks land wherever a slot is free first, not rank by
//     rank, so no skew: 256 x 8192 35.5 (skew 0.3: 40.1), 384 x 4096 26.9 (29.6), 1024 x 1024 19.7 (20.4).
static MarchModel march_model(int prec, bool gpbc, long long nodes) {
    if (prec == LB_PREC_BF16)
        return gpbc ? MarchModel{0.16, 1.4, true} : MarchModel{march_dependent(prec, gpbc, nodes) ? 0.0 : 0.30, 1.15, true};
    return {0.08, gpbc ? 1.6 : 1.2, true};
}

// The row-march variant of a handle: f(stress mode, boundary, scheme, strips) as constants.
template <int V> using Num = std::integral_constant<int, V>;
template <typename F>
auto march_variant(const lb_handle* h, F&& f) {
    auto with_strip = [&](auto sm, auto bnd, auto sch) {
        if (h->march_strip == kOdd) return f(sm, bnd, sch, Num<kOdd>{});
        return h->march_strip == kPart ? f(sm, bnd, sch, Num<kPart>{}) : f(sm, bnd, sch, Num<kFull>{});
    };
    auto with_mode = [&](auto bnd, auto sch) {
        return h->smode ? with_strip(Num<1>{}, bnd, sch) : with_strip(Num<0>{}, bnd, sch);
    };
    if (h->scheme == 1) return with_strip(Num<0>{}, Num<0>{}, Num<1>{});
    if (h->scheme == 3) return with_mode(Num<0>{}, Num<3>{});
    if (h->gpbc) return with_mode(Num<1>{}, Num<0>{});
    if (h->moving) return with_mode(Num<2>{}, Num<0>{});
    return with_mode(Num<0>{}, Num<0>{});
}

// Whole strips always march, which makes small ones slower than they need be in FP32; other widths where that is the faster
// kernel.  A march step lasts 7 us at least (a chain of rows), a tile step 4, but the tile kernel takes 1.3 to 2
// times as long per node.  Tile / march, us: FP32 128 x 16 3.9 / 7.1, 128 x 512 5.4 / 7.6, 1024 x 128 7.8 / 9.3, 512 x
// 512 11.7 / 10.7, 100 x 1600 10.1 / 12.7, 200 x 1600 15.8 / 16.8, 500 x 800 17.5 / 16.8, 1000 x 777 30.1 / 23.0, 2049 x 600
// 52.3 / 35.0; BF16 128 x 16 7.2 / 7.0, 512 x 512 15.5 / 10.0, 200 x 400 9.4 / 10.6, 70 x 2000 16.2 / 15.7, 100 x 1600 16.0 /
// 13.3, 1000 x 300 18.1 / 13.5, 1001 x 777 44.8 / 26.8.  Below 96 columns half of a strip's threads have none.
static bool march_pays(const lb_handle* h) {
    if (h->nx % kMarchW == 0) return true;
    return h->nx >= 96 && march_strip_width(h->nx) > 0 && (long long)h->nx * h->ny[0] >= (h->prec == LB_PREC_BF16 ? 150000 : 400000);
}

lb_status plan_march(lb_handle* h) {
    h->march = false;
    if (h->n_ch != 1 || (h->prec != LB_PREC_F32 && h->prec != LB_PREC_BF16) || h->ny[0] < 16 ||
        (h->flags & LB_GRID_TILE_ONLY) || h->scheme == 2 || (h->scheme == 3 && (h->gpbc || h->moving)) || !march_pays(h))
        return LB_OK;
    h->march_strip = h->nx % kMarchW == 0 ? kFull : (h->nx % (h->prec == LB_PREC_BF16 ? 8 : 4) == 0 ? kPart : kOdd);
    if (h->march_strip == kOdd && (long long)h->nx * (h->ny[0] + 4) >= (1ll << 31) - 4096) return LB_OK;  // (copy coordinates)
    if (!make_pop_map(h, h->popA, &h->mapA) || !make_pop_map(h, h->popB, &h->mapB)) return LB_OK;
    h->mapA_buf = h->popA;
    h->mapB_buf = h->popB;
    int bps = 0, nsm = 0;
    cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->dev);
    if (e == cudaSuccess)
        e = march_variant(h, [&](auto sm, auto bnd, auto sch, auto strip) {
            constexpr int SM = decltype(sm)::value, B = decltype(bnd)::value, S = decltype(sch)::value;
            return h->prec == LB_PREC_F32 ? march_occupancy<float, float, SM, B, S, decltype(strip)::value>(&bps)
                                          : march_occupancy<__nv_bfloat16, float, SM, B, S, decltype(strip)::value>(&bps);
        });
    if (e != cudaSuccess) return cuda_fail(e, "lb_create: march occupancy");
    if (bps < 1) return LB_OK;
    const int slots = bps * nsm;
    const std::vector<MarchItem> items = short_items(
        fine_items(march_plan(h->nx, h->ny[0], bps, nsm, march_model(h->prec, h->gpbc, h->nodes)), h->nx, h->ny[0], slots), h->nx);
    LB_CK(cudaMalloc(&h->march_items_d, sizeof(MarchItem) * items.size()));
    LB_CK(cudaMemcpyAsync(h->march_items_d, items.data(), sizeof(MarchItem) * items.size(), cudaMemcpyHostToDevice, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));  // (the host copy goes)
    h->n_march_items = (int)items.size();
    if ((int)h->items.size() < h->n_march_items) {  // the partials buffer serves both plans
        cudaFree(h->partials);
        h->partials = nullptr;
        LB_CK(cudaMalloc(&h->partials, 4 * sizeof(double) * h->n_march_items));
    }
    h->march_grid = std::min(h->n_march_items, slots);
    h->march = true;
    return LB_OK;
}

lb_status validate(const lb_grid* g, const lb_params* p, const lb_boundary* b) {
    if (!g || !p || !b) return fail(LB_EINVAL, "lb_create: null argument%s");
    if (g->n_channels < 1 || g->nx < 1 || !g->ny) return fail(LB_EINVAL, "lb_create: need n_channels >= 1, nx >= 1, ny%s");
    if (g->precision < 0 || g->precision > 4) return fail(LB_EINVAL, "lb_create: unknown precision%s");
    if (g->stress_mode < 0 || g->stress_mode > 1) return fail(LB_EINVAL, "lb_create: unknown stress_mode%s");
    if ((b->walls != LB_WALLS_BOUNCE_BACK && b->walls != LB_WALLS_COUETTE) ||
        (b->x_mode != LB_X_PERIODIC && b->x_mode != LB_X_GPBC))
        return fail(LB_EINVAL, "lb_create: walls must be LB_WALLS_BOUNCE_BACK or LB_WALLS_COUETTE and x_mode LB_X_PERIODIC or LB_X_GPBC%s");
    const bool gn = (g->flags & LB_GRID_GENERALIZED_NEWTONIAN) != 0, dv = (g->flags & LB_GRID_STRESS_DIVERGENCE) != 0;
    const bool rx = (g->flags & LB_GRID_RELAXATION_MODEL) != 0;
    if ((int)gn + (int)dv + (int)rx > 1)
        return fail(LB_EINVAL, "lb_create: choose one comparison scheme, or the relaxation-time extensions%s");
    if (rx && g->precision != LB_PREC_F64 && g->precision != LB_PREC_F32 && g->precision != LB_PREC_BF16)
        return fail(LB_EINVAL, "lb_create: the relaxation-time extensions run in FP64, FP32 or BF16%s");
    if ((gn || dv) && (g->stress_mode != 0 || b->walls != LB_WALLS_BOUNCE_BACK || b->x_mode != LB_X_PERIODIC))
        return fail(LB_EINVAL, "lb_create: the comparison schemes run with stress mode 0, periodic x and bounce-back walls%s");
    if ((gn || dv) && g->precision != LB_PREC_F64 && g->precision != LB_PREC_F32 && g->precision != LB_PREC_BF16)
        return fail(LB_EINVAL, "lb_create: the comparison schemes run in FP64, FP32 or BF16%s");
    for (int c = 0; c < g->n_channels; ++c) {
        if (g->ny[c] < 3) return fail(LB_EINVAL, "lb_create: ny must be >= 3%s");
        if ((long long)g->ny[c] * g->nx > (1ll << 40)) return fail(LB_EINVAL, "lb_create: channel too large%s");
        const lb_params& q = p[c];
        const double v[8] = {q.tau_lb, q.g_x, q.G_inf, q.tau0, q.theta, q.rho0, q.rho_pert_amp, 0.0};
        for (double x : v)
            if (std::isnan(x) || std::isinf(x)) return fail(LB_EINVAL, "lb_create: non-finite parameter%s");
        if (!(q.tau_lb > 0.5)) return fail(LB_EINVAL, "lb_create: tau_lb must be > 1/2%s");
        if (q.G_inf < 0 || q.tau0 < 0 || q.theta < 0) return fail(LB_EINVAL, "lb_create: G_inf, tau0, theta must be >= 0%s");
        if (!(q.gamma_c > 0)) return fail(LB_EINVAL, "lb_create: gamma_c must be > 0 (inf allowed)%s");
        if (!(q.rho0 > 0) || q.rho_pert_amp < 0 || q.rho_pert_amp >= 1)
            return fail(LB_EINVAL, "lb_create: need rho0 > 0 and 0 <= rho_pert_amp < 1%s");
    }
    return LB_OK;
}

template <typename T>
void free_dev(T*& p) {
    if (p) cudaFree((void*)p);
    p = nullptr;
}

void release(lb_handle* h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    free_dev(h->popA); free_dev(h->popB); free_dev(h->drho); free_dev(h->sig3); free_dev(h->sig4); free_dev(h->snn); free_dev(h->phi);
    free_dev(h->uprev); free_dev(h->chan); free_dev(h->items_d); free_dev(h->item_begin_d);
    free_dev(h->partials); free_dev(h->mon_d); free_dev(h->status_d); free_dev(h->base_d); free_dev(h->P_d);
    free_dev(h->node_off_d); free_dev(h->ny_d); free_dev(h->gx_d); free_dev(h->fields[0]); free_dev(h->fields[1]);
    free_dev(h->hstage);
    free_dev(h->ws_prm); free_dev(h->ws_row_off); free_dev(h->ws_rows); free_dev(h->ws_grid); free_dev(h->ws_scale);
    free_dev(h->march_items_d);
    free_dev(h->sweep_steps_d);
    free_dev(h->sweep_res_d);
    free_dev(h->sweep_order_d);
    free_dev(h->gcol);
    free_dev(h->gpart);
    free_dev(h->gcount);
    free_dev(h->done_count_d);
    if (h->status_h) cudaFreeHost(h->status_h);
    if (h->mon_h) cudaFreeHost(h->mon_h);
    if (h->status_ev) cudaEventDestroy(h->status_ev);
    for (int k = 0; k < 2; ++k)
        if (h->gexec[k]) cudaGraphExecDestroy(h->gexec[k]);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    for (cudaStream_t q : h->gstreams) cudaStreamDestroy(q);
    for (cudaEvent_t q : h->gevents) cudaEventDestroy(q);
    if (h->fork_ev) cudaEventDestroy(h->fork_ev);
    if (h->sweep_gexec) cudaGraphExecDestroy(h->sweep_gexec);
    delete h;
}

lb_status ensure_hstage(lb_handle* h, size_t bytes) {
    if (h->hstage_bytes >= bytes) return LB_OK;
    free_dev(h->hstage);
    h->hstage_bytes = 0;
    LB_CK(cudaMalloc(&h->hstage, bytes));
    h->hstage_bytes = bytes;
    return LB_OK;
}

// Key of the stochastic rounding for one step (SplitMix64 finaliser of the handle seed and step).
uint32_t step_key(const lb_handle* h, long long step) {
    uint64_t z = h->params[0].seed + 0x632BE59BD9B4E019ull + (uint64_t)step * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)(z ^ (z >> 31));
}

template <typename T, typename C>
StepArgs<T, C> base_args(lb_handle* h) {
    StepArgs<T, C> a{};
    a.pin = (const T*)h->popA;
    a.pout = (T*)h->popB;
    a.drho = (C*)h->drho;
    a.sig3 = (C*)h->sig3;
    a.sig4 = (C*)h->sig4;
    a.uprev = (C*)h->uprev;
    a.snn = (C*)h->snn;
    a.phi = (double*)h->phi;
    a.partials = h->partials;
    a.items = h->items_d;
    a.chan = (const ChanParams<C>*)h->chan;
    a.status = h->status_d;
    a.nx = h->nx;
    a.guard = (C)kGuard;
    a.gcol = (const C*)h->gcol;
    a.gny = h->gny;
    return a;
}

// A body force or (WALL) wall velocity of one channel, or all (-1): host -> channel table, stream-ordered, by value.
template <bool WALL>
lb_status push_drive(lb_handle* h, int channel, double v) {
    const int c0 = std::max(channel, 0), n = channel < 0 ? h->n_ch : 1;
    const int threads = std::min(kDriveThreads, (n + 31) / 32 * 32), grid = (n + kDriveThreads - 1) / kDriveThreads;
    if (h->csize == 8)
        LB_CK(launch_dependent(true, k_apply_drive<double, WALL>, grid, threads, 0, h->stream, (ChanParams<double>*)h->chan, h->gx_d, v, c0, n, h->n_ch, h->nx));
    else
        LB_CK(launch_dependent(true, k_apply_drive<float, WALL>, grid, threads, 0, h->stream, (ChanParams<float>*)h->chan, h->gx_d, v, c0, n, h->n_ch, h->nx));
    return LB_OK;
}

// Under GPBC every step kernel needs the boundary columns of its input buffer.
template <typename T, typename C>
cudaError_t gpbc_columns(lb_handle* h) {
    if (!h->gpbc) return cudaSuccess;
    return launch_gpbc_columns<T, C>((const T*)h->popA, (const ChanParams<C>*)h->chan, (C*)h->gcol, h->n_ch, h->nx,
                                     h->gny, h->gpbc_max_ny, h->gpart, h->gcount, h->stream);
}

// The comparison schemes are instantiated for the three main precisions (T and C of one type, or
// BF16 storage with FP32 arithmetic); lb_create refuses them with the mixed diagnostic ones.
template <typename T, typename C>
constexpr bool kSchemeTypes = std::is_same<T, C>::value || std::is_same<T, __nv_bfloat16>::value;

template <typename T, typename C>
cudaError_t launch(lb_handle* h, const StepArgs<T, C>& a) {
    const int n = (int)h->items.size();
    if constexpr (kSchemeTypes<T, C>) {
        if (h->scheme == 3)
            return h->smode == 0 ? launch_step_tile<T, C, 0, 3>(a, n, h->smem, h->stream)
                                 : launch_step_tile<T, C, 1, 3>(a, n, h->smem, h->stream);
        if (h->scheme == 1) return launch_step_tile<T, C, 0, 1>(a, n, h->smem, h->stream);
        if (h->scheme == 2) {
            // stress divergence: Sigma^nN of every node of this step first, then the step (or the
            // fields pass) that differentiates it
            StepArgs<T, C> s = a;
            s.flags = F_SNN;
            cudaError_t e = launch_step_tile<T, C, 0, 2>(s, n, h->smem, h->stream);
            if (e != cudaSuccess) return e;
            StepArgs<T, C> b = a;
            b.flags |= F_DIV;
            return launch_step_tile<T, C, 0, 2>(b, n, h->smem, h->stream);
        }
    } else {
        if (h->scheme != 0) return cudaErrorNotSupported;
    }
    if (h->smode == 0) return launch_step_tile<T, C, 0>(a, n, h->smem, h->stream);
    return launch_step_tile<T, C, 1>(a, n, h->smem, h->stream);
}

// The row-march kernel's last CTA mirrors the status word into mapped host memory every step and,
// on monitor steps (F_RESID / F_MON), reduces the item partials into mon_d.
void march_monitor(lb_handle* h, int flags, MarchCtl& ctl) {
    const bool mon = (flags & (F_RESID | F_MON)) != 0;
    ctl.done_count = h->done_count_d;
    ctl.status_host = h->status_hd;
    ctl.mon = mon ? (double*)h->mon_d : nullptr;
    ctl.state_index = h->step;
    ctl.with_residual = (flags & F_RESID) ? 1 : 0;
}

// The row-march kernel: a step, or (F_FIELDS) the fields of the stored state.
template <typename T, bool FIELDS>
cudaError_t launch_march_as(lb_handle* h, const StepArgs<T, float>& a) {
    // (the fields pass has its own wait limit: lb_set_wait_limit speaks of steps)
    MarchCtl ctl{h->march_items_d, h->n_march_items, h->status_d, h->P[0], h->base[0], FIELDS ? kDefaultWaitNs : h->wait_ns};
    march_monitor(h, a.flags, ctl);
    ctl.dependent = march_dependent(h->prec, h->gpbc, h->nodes);
    const CUtensorMap& m = ((const void*)a.pin == h->mapA_buf) ? h->mapA : h->mapB;
    return march_variant(h, [&](auto sm, auto bnd, auto sch, auto strip) {
        return launch_step_march<T, float, decltype(sm)::value, decltype(bnd)::value, decltype(sch)::value, FIELDS,
                                 decltype(strip)::value>(m, a, ctl, h->march_grid, h->stream);
    });
}
template <typename T, typename C>
cudaError_t launch_march(lb_handle* h, const StepArgs<T, C>& a) {
    if constexpr (std::is_same<C, float>::value && (std::is_same<T, float>::value || std::is_same<T, __nv_bfloat16>::value))
        return (a.flags & F_FIELDS) ? launch_march_as<T, true>(h, a) : launch_march_as<T, false>(h, a);
    else
        return cudaErrorNotSupported;
}

// The resident kernel of a handle's types and thread count: f(stress mode, NT) as constants.
template <typename T, typename F>
cudaError_t resident_variant(const lb_handle* h, int threads, F&& f) {
    auto with_mode = [&](auto nt) { return h->smode ? f(Num<1>{}, nt) : f(Num<0>{}, nt); };
    if constexpr (std::is_same<T, double>::value) {
        return with_mode(Num<128>{});
    } else {
        if (threads <= 128) return with_mode(Num<128>{});
        if (threads <= 320) return with_mode(Num<320>{});
        return with_mode(Num<640>{});
    }
}
template <typename T, typename C>
constexpr bool kResidentTypes = std::is_same<T, C>::value || std::is_same<T, __nv_bfloat16>::value;

// Whether runs of plain steps of this handle stay on chip (lb_step_resident.cuh): one channel of the paper's
// scheme that a cluster can hold with one node per thread, and where that is the faster way.
void plan_resident(lb_handle* h) {
    h->res_cl = 0;
    if (h->n_ch != 1 || h->march || h->scheme != 0 || h->gpbc || (h->flags & (LB_GRID_TILE_ONLY | LB_GRID_NO_GRAPH)) ||
        ((h->flags & LB_GRID_BF16_STOCHASTIC) && h->prec == LB_PREC_BF16))
        return;
    const int nx = h->nx, ny = h->ny[0];
    with_types(h->prec, [&](auto tt, auto tc) {
        LB_TYPES(tt, tc);
        if constexpr (kResidentTypes<T, C>) {
            const int most = std::is_same<T, double>::value ? 128 : 640;  // threads of a CTA, see lb_step_resident.cuh
            for (int cl : {16, 8, 4, 2, 1}) {
                if (ny / cl < 2 || (long long)nx * ny > 1 << 20) continue;
                const int threads = resident_threads(ny, nx, cl);
                const size_t smem = resident_smem<T, C>(ny, nx, cl);
                if (threads > most || smem > 227 * 1024) continue;
                int clusters = 0;
                const cudaError_t e = resident_variant<T>(h, threads, [&](auto sm, auto nt) {
                    return resident_capacity<T, C, decltype(sm)::value, decltype(nt)::value>(cl, threads, smem, &clusters);
                });
                if (e != cudaSuccess) (void)cudaGetLastError();
                if (e != cudaSuccess || clusters < 1) continue;
                h->res_cl = cl;
                h->res_threads = threads;
                h->res_smem = smem;
                break;
            }
        }
        return 0;
    });
}

constexpr int kGraphSteps = 32;  // steps per captured graph (even)

// Capture kGraphSteps plain steps (no velocity save, no residual, no stochastic rounding) starting
// from the current input buffer on the handle's private capture stream.
template <typename T, typename C>
lb_status capture_graph(lb_handle* h, int slot) {
    if (!h->cap_stream) LB_CK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    if (h->gexec[slot]) {
        LB_CK(cudaGraphExecDestroy(h->gexec[slot]));
        h->gexec[slot] = nullptr;
        h->gexec_pin[slot] = nullptr;
    }
    const void* pin = h->popA;
    cudaStream_t user = h->stream;
    h->stream = h->cap_stream;
    cudaError_t e = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        h->stream = user;
        return cuda_fail(e, "graph capture begin");
    }
    for (int k = 0; k < kGraphSteps && e == cudaSuccess; ++k) {
        StepArgs<T, C> a = base_args<T, C>(h);
        a.flags = (h->flags & LB_GRID_STORE_SIGMA) ? F_STORE_SIGMA : 0;
        e = gpbc_columns<T, C>(h);
        if (e == cudaSuccess) e = launch<T, C>(h, a);
        std::swap(h->popA, h->popB);
    }
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(h->cap_stream, &g);
    h->stream = user;
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&h->gexec[slot], g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        h->gexec[slot] = nullptr;
        return cuda_fail(e, "graph capture");
    }
    h->gexec_pin[slot] = pin;
    return LB_OK;
}

template <typename T, typename C>
lb_status run_steps(lb_handle* h, long n) {
    const bool sr = (h->flags & LB_GRID_BF16_STOCHASTIC) && h->prec == LB_PREC_BF16;
    long s = 1;
    // A small single channel takes its plain steps on chip, many per launch (the last two of the call, with the
    // velocity save and the residual, follow one by one); at least kResidentSteps, since a launch costs the time
    // of a few steps, at most 65536, so that no launch lasts longer than a fraction of a second.
    if (h->res_cl > 0) {
        if constexpr (kResidentTypes<T, C>) {
            while (n - s + 1 >= kResidentSteps + 2) {
                const long run = std::min(n - s + 1 - 2, 65536L);
                StepArgs<T, C> a = base_args<T, C>(h);
                a.flags = (h->flags & LB_GRID_STORE_SIGMA) ? F_STORE_SIGMA : 0;
                LB_CK((resident_variant<T>(h, h->res_threads, [&](auto sm, auto nt) {
                    return launch_step_resident<T, C, decltype(sm)::value, decltype(nt)::value>(
                        a, (T*)h->popA, run, h->res_cl, h->res_threads, h->res_smem, h->stream);
                })));
                h->step += run;
                s += run;
            }
        }
    }
    // Runs of plain steps replay a captured graph; the last two steps of the call (velocity save,
    // residual) are always launched one by one.
    if (!h->march && h->res_cl == 0 && !sr && !(h->flags & LB_GRID_NO_GRAPH)) {
        while (n - s + 1 >= kGraphSteps + 2) {
            int slot = h->gexec_pin[0] == h->popA ? 0 : (h->gexec_pin[1] == h->popA ? 1 : -1);
            if (slot < 0) {
                slot = h->gexec_pin[0] ? 1 : 0;
                lb_status st = capture_graph<T, C>(h, slot);
                if (st != LB_OK) return st;
            }
            LB_CK(cudaGraphLaunch(h->gexec[slot], h->stream));
            ++h->graph_replays;
            h->step += kGraphSteps;
            s += kGraphSteps;
        }
    }
    for (; s <= n; ++s) {
        StepArgs<T, C> a = base_args<T, C>(h);
        int f = 0;
        if (h->flags & LB_GRID_STORE_SIGMA) f |= F_STORE_SIGMA;
        if (sr) f |= F_SR;
        a.sr_key = step_key(h, h->step);
        bool resid = false, mon = false;
        if (h->monitor_mode == LB_MONITOR_FLUX_MAX) {
            mon = (s == n);  // flux and max |u| of the last step's state: no saved velocity
            if (mon) f |= F_MON;
        } else {
            resid = mon = (s == n) && (h->uprev_state == h->step - 1);
            if (s >= n - 1) f |= F_SAVE_U;
            if (resid) f |= F_RESID;
        }
        a.flags = f;
        LB_CK((gpbc_columns<T, C>(h)));
        if (h->march) LB_CK((launch_march<T, C>(h, a)));
        else LB_CK((launch<T, C>(h, a)));
        if (mon) {
            if (!h->march) {  // (the row-march kernel's last CTA reduces its partials itself)
                k_reduce_residual<<<h->n_ch, 32, 0, h->stream>>>(h->partials, h->item_begin_d, h->status_d, h->mon_d,
                                                                 h->nx, h->step, resid ? 1 : 0);
                LB_CK(cudaGetLastError());
            }
            h->mon_state = h->step;
            h->mon_resid = resid;
        }
        if (f & F_SAVE_U) h->uprev_state = h->step;
        std::swap(h->popA, h->popB);
        ++h->step;
    }
    return LB_OK;
}

// The fields of the current state into device buffers (any may be null; 16-byte aligned) of type double (out64)
// or float.
lb_status fields_pass(lb_handle* h, void* fu, void* fs, void* fr, bool out64) {
    return with_types(h->prec, [&](auto tt, auto tc) -> lb_status {
        LB_TYPES(tt, tc);
        StepArgs<T, C> a = base_args<T, C>(h);
        a.flags = F_FIELDS | (out64 ? F_OUT64 : 0);
        a.fu = fu;
        a.fsig = fs;
        a.frho = fr;
        LB_CK((gpbc_columns<T, C>(h)));
        if (h->march) LB_CK((launch_march<T, C>(h, a)));
        else LB_CK((launch<T, C>(h, a)));
        return LB_OK;
    });
}

// The handle's staging buffer of 7 values per node (u, sigma, rho one after the other), of float or double.
lb_status ensure_fields(lb_handle* h, size_t value_size) {
    void*& f = h->fields[value_size == 8];
    if (!f) LB_CK(cudaMalloc(&f, 7 * (size_t)h->nodes * value_size + 64));
    return LB_OK;
}
// its parts, each on a 16-byte boundary
struct FieldParts {
    char *u, *sigma, *rho;
};
FieldParts field_parts(lb_handle* h, size_t value_size) {
    char* b = (char*)h->fields[value_size == 8];
    const size_t n = (size_t)h->nodes * value_size;
    return FieldParts{b, b + (2 * n + 15) / 16 * 16, b + (2 * n + 15) / 16 * 16 + 4 * n};
}

lb_status poll_status(lb_handle* h, bool wait) {
    if (h->march) {  // the row-march kernel stores the status word into mapped host memory itself
        const int s = *(volatile const int*)h->status_h;
        if (s & 1) h->any_unstable = true;
        if (s & 2) h->any_timeout = true;
        return LB_OK;
    }
    if (h->status_pending) {
        cudaError_t q = wait ? cudaEventSynchronize(h->status_ev) : cudaEventQuery(h->status_ev);
        if (q == cudaSuccess) {
            h->status_pending = false;
            for (int c = 0; c < h->n_ch; ++c) {
                if (h->status_h[c] & 1) h->any_unstable = true;
                if (h->status_h[c] & 2) h->any_timeout = true;
            }
        } else if (q != cudaErrorNotReady) {
            return cuda_fail(q, "status event");
        }
    }
    return LB_OK;
}

lb_status request_status(lb_handle* h) {
    LB_CK(cudaMemcpyAsync(h->status_h, h->status_d, sizeof(int) * h->n_ch, cudaMemcpyDeviceToHost, h->stream));
    LB_CK(cudaEventRecord(h->status_ev, h->stream));
    h->status_pending = true;
    return LB_OK;
}

constexpr int kSweepNPT = 4;  // nodes per thread of the sweep kernel

// Channels of one width class (floor(log2 ny)) run in their own persistent launch with their own
// tuned configuration; the classes' launches run side by side on forked streams.
int width_class(int ny) {
    int k = 0;
    while ((2 << k) <= ny) ++k;
    return k;
}
bool sweep_fits(int ny_max, int nx, int nt, int cl) {
    const int rows = (ny_max + cl - 1) / cl;
    return (long long)rows * nx <= (long long)nt * kSweepNPT;
}
size_t sweep_smem(const lb_handle* h, int ny_max, int cl) {
    const int rows = (ny_max + cl - 1) / cl + 4;
    return (size_t)rows * h->nx * 2 * h->csize;
}
// Shared-memory resident variant: every CTA owns >= 3 rows (halo rows come from the neighbours),
// and its rows, halos and velocity rows fit the 227 KB of one CTA.
size_t sweep_smem_resident(const lb_handle* h, int ny_max, int cl) {
    const int rows = (ny_max + cl - 1) / cl;
    if (h->csize == 4) return h->tsize == 2 ? sweep_pair_smem<__nv_bfloat16>(rows, h->nx) : sweep_pair_smem<float>(rows, h->nx);
    return sweep_smem_bytes<double, double>(rows, h->nx);
}
bool sweep_config_fits(const lb_handle* h, const SweepGroup& g, int var, int nt, int cl) {
    if (cl < 1 || cl > 16 || (nt != 128 && nt != 256) || !sweep_fits(g.ny_max, h->nx, nt, cl)) return false;
    if (var == 0) return sweep_smem(h, g.ny_max, cl) <= 200 * 1024;
    return g.ny_min / cl >= 3 && sweep_smem_resident(h, g.ny_max, cl) <= 227 * 1024;
}

// Threads and width of a resident sweep kernel as constants.
template <typename F>
cudaError_t sweep_variant(const lb_handle* h, int nt, F&& f) {
    if (h->nx == 4) return nt == 128 ? f(Num<128>{}, Num<4>{}) : f(Num<256>{}, Num<4>{});
    return nt == 128 ? f(Num<128>{}, Num<0>{}) : f(Num<256>{}, Num<0>{});
}

template <typename T, typename C>
cudaError_t sweep_launch(lb_handle* h, const SweepGroup& g, int var, int nt, int cl, double tol, int check,
                         long long max_steps, cudaStream_t stream) {
    SweepArgs<T, C> a{};
    a.popA = (T*)h->popA;
    a.popB = (T*)h->popB;
    a.drho = (C*)h->drho;
    a.uprev = (C*)h->uprev;
    a.chan = (const ChanParams<C>*)h->chan;
    a.status = h->status_d;
    a.order = h->sweep_order_d + g.begin;
    a.steps_out = h->sweep_steps_d;
    a.res_out = h->sweep_res_d;
    a.nx = h->nx;
    a.check = check;
    a.max_steps = max_steps;
    a.tol = tol;
    a.sr = (h->flags & LB_GRID_BF16_STOCHASTIC) && h->prec == LB_PREC_BF16;
    a.sr_key = step_key(h, h->step + 0x5bd1e995ll);
    if (var == 1) {
        const size_t smem = sweep_smem_resident(h, g.ny_max, cl);
        return sweep_variant(h, nt, [&](auto threads, auto width) {  // (4 columns: width known at compile time)
            constexpr int NT = decltype(threads)::value, NX = decltype(width)::value;
            if constexpr (std::is_same<C, float>::value) return launch_sweep_pair<T, NT, kSweepPairs, NX>(a, g.count, cl, smem, stream);
            else return launch_sweep_smem<T, C, NT, kSweepNPT, NX>(a, g.count, cl, smem, stream);
        });
    }
    const size_t smem = sweep_smem(h, g.ny_max, cl);
    if (h->nx == 4) {
        if (nt == 128) return launch_sweep<T, C, 128, kSweepNPT, 4>(a, g.count, cl, smem, stream);
        return launch_sweep<T, C, 256, kSweepNPT, 4>(a, g.count, cl, smem, stream);
    }
    if (nt == 128) return launch_sweep<T, C, 128, kSweepNPT>(a, g.count, cl, smem, stream);
    return launch_sweep<T, C, 256, kSweepNPT>(a, g.count, cl, smem, stream);
}

cudaError_t sweep_launch_any(lb_handle* h, const SweepGroup& g, int var, int nt, int cl, double tol, int check,
                             long long max_steps, cudaStream_t stream) {
    return with_types(h->prec, [&](auto tt, auto tc) -> cudaError_t {
        LB_TYPES(tt, tc);
        if constexpr (std::is_same<T, double>::value != std::is_same<C, double>::value) return cudaErrorNotSupported;
        else return sweep_launch<T, C>(h, g, var, nt, cl, tol, check, max_steps, stream);
    });
}

// Clusters of this configuration the device can hold at once (0: never launched).
int sweep_capacity(lb_handle* h, const SweepGroup& g, int var, int nt, int cl) {
    int n = 0;
    const cudaError_t e = with_types(h->prec, [&](auto tt, auto tc) -> cudaError_t {
        LB_TYPES(tt, tc);
        if constexpr (std::is_same<T, double>::value != std::is_same<C, double>::value) return cudaErrorNotSupported;
        else {
            if (var == 1) {
                const size_t smem = sweep_smem_resident(h, g.ny_max, cl);
                return sweep_variant(h, nt, [&](auto threads, auto width) {
                    constexpr int NT = decltype(threads)::value, NX = decltype(width)::value;
                    if constexpr (std::is_same<C, float>::value) return launch_sweep_pair_capacity<T, NT, kSweepPairs, NX>(cl, smem, &n);
                    else return launch_sweep_smem_capacity<T, C, NT, kSweepNPT, NX>(cl, smem, &n);
                });
            }
            const size_t smem = sweep_smem(h, g.ny_max, cl);
            if (h->nx == 4)
                return nt == 128 ? launch_sweep_capacity<T, C, 128, kSweepNPT, 4>(cl, smem, &n)
                                 : launch_sweep_capacity<T, C, 256, kSweepNPT, 4>(cl, smem, &n);
            return nt == 128 ? launch_sweep_capacity<T, C, 128, kSweepNPT>(cl, smem, &n)
                             : launch_sweep_capacity<T, C, 256, kSweepNPT>(cl, smem, &n);
        }
    });
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}

// Stable channels, widest first (the longest-running clusters start first), split into width
// classes; a class keeps the configuration it was tuned (or set) with.
lb_status sweep_order(lb_handle* h, int* n_active, const std::vector<char>* only = nullptr) {
    std::vector<int> st(h->n_ch);
    LB_CK(cudaMemcpyAsync(st.data(), h->status_d, sizeof(int) * h->n_ch, cudaMemcpyDeviceToHost, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    std::vector<int> order;
    for (int c = 0; c < h->n_ch; ++c)
        if (st[c] == 0 && (!only || (*only)[c])) order.push_back(c);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return h->ny[a] > h->ny[b]; });
    if (!h->sweep_order_d) {
        LB_CK(cudaMalloc(&h->sweep_order_d, sizeof(int) * h->n_ch));
        LB_CK(cudaMalloc(&h->sweep_steps_d, sizeof(long long) * h->n_ch));
        LB_CK(cudaMalloc(&h->sweep_res_d, sizeof(double) * h->n_ch));
    }
    if (!order.empty())
        LB_CK(cudaMemcpyAsync(h->sweep_order_d, order.data(), sizeof(int) * order.size(), cudaMemcpyHostToDevice, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));  // (the host copy goes)
    std::vector<SweepGroup> groups;
    for (int k = 0; k < (int)order.size(); ++k) {
        const int ny = h->ny[order[k]];
        if (groups.empty() || width_class(ny) != groups.back().cls) {
            SweepGroup g;
            g.cls = width_class(ny);
            g.begin = k;
            g.ny_max = ny;
            for (const SweepGroup& old : h->sweep_groups)
                if (old.cls == g.cls) { g.var = old.var; g.nt = old.nt; g.cl = old.cl; g.tune_ms = old.tune_ms; }
            groups.push_back(g);
        }
        groups.back().count += 1;
        groups.back().ny_min = ny;
    }
    for (SweepGroup& g : groups) {
        // a kept configuration must still fit (it does when channels only leave); a class that has
        // lost half of its channels is tuned again (few clusters: the timing becomes per-step
        // latency instead of throughput), unless the configuration was fixed by the caller
        if (g.nt && !sweep_config_fits(h, g, g.var, g.nt, g.cl)) g.nt = 0;
        for (const SweepGroup& old : h->sweep_groups)
            if (old.cls == g.cls && g.nt && !h->sweep_fixed && 2 * g.count <= old.count) g.nt = 0;
    }
    h->sweep_groups = groups;
    *n_active = (int)order.size();
    return LB_OK;
}

// Autotuner: per width class, time a short sweep of that class alone (no channel can converge:
// tol < 0) for every (kernel, threads, cluster size) that fits, from the same saved state, and
// keep the fastest.  The state is restored.
lb_status sweep_tune(lb_handle* h, bool all) {
    const size_t pop_b = 9 * h->planes * h->tsize, dr_b = h->planes * h->csize, up_b = 2 * h->planes * h->csize;
    void* save = nullptr;
    LB_CK(cudaMalloc(&save, pop_b + dr_b + up_b));
    char* sv = (char*)save;
    auto restore = [&]() -> cudaError_t {
        cudaError_t e = cudaMemcpyAsync(h->popA, sv, pop_b, cudaMemcpyDeviceToDevice, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(h->drho, sv + pop_b, dr_b, cudaMemcpyDeviceToDevice, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(h->uprev, sv + pop_b + dr_b, up_b, cudaMemcpyDeviceToDevice, h->stream);
        return e;
    };
    cudaError_t e = cudaMemcpyAsync(sv, h->popA, pop_b, cudaMemcpyDeviceToDevice, h->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sv + pop_b, h->drho, dr_b, cudaMemcpyDeviceToDevice, h->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sv + pop_b + dr_b, h->uprev, up_b, cudaMemcpyDeviceToDevice, h->stream);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    bool none = false;
    for (SweepGroup& g : h->sweep_groups) {
        if (e != cudaSuccess) break;
        if (g.nt && !all) continue;
        double best = 1e300;
        for (int var : {0, 1})
            for (int nt : {128, 256})
                for (int cl : {1, 2, 4, 8, 16}) {
                    if (e != cudaSuccess || !sweep_config_fits(h, g, var, nt, cl)) continue;
                    if (sweep_capacity(h, g, var, nt, cl) < 1) continue;  // cannot be co-scheduled
                    float ms = 0.f;
                    bool launched = true;
                    for (int rep = 0; rep < 2 && e == cudaSuccess && launched; ++rep) {  // first run warms up
                        e = restore();
                        if (e == cudaSuccess) e = cudaEventRecord(e0, h->stream);
                        if (e == cudaSuccess) {
                            // a cluster shape the device cannot co-schedule is refused at launch (a
                            // configuration error that leaves the context usable): skip it
                            const cudaError_t le = sweep_launch_any(h, g, var, nt, cl, -1.0, 16, 256, h->stream);
                            if (le != cudaSuccess) {
                                launched = false;
                                (void)cudaGetLastError();
                            }
                        }
                        if (e == cudaSuccess) e = cudaEventRecord(e1, h->stream);
                        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                    }
                    if (e == cudaSuccess && launched && ms < best) {
                        best = ms;
                        g.var = var;
                        g.nt = nt;
                        g.cl = cl;
                        g.tune_ms = ms;
                    }
                }
        if (best == 1e300) none = true;
    }
    if (e == cudaSuccess) e = restore();
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(save);
    if (e != cudaSuccess || none) {
        for (SweepGroup& g : h->sweep_groups) g.nt = 0;
        if (e != cudaSuccess) return cuda_fail(e, "lb_run_until_steady: autotune");
        return fail(LB_ECUDA, "lb_run_until_steady: a channel is too wide for the sweep kernels, or no configuration could be launched%s");
    }
    return LB_OK;
}

// One persistent launch per width class on forked streams, joined back: captured once as a CUDA
// graph (on the handle's private capture stream) and replayed while the arguments, the class
// configurations and the population buffer that holds the state (lb_step swaps the two) stay the same.
lb_status sweep_run(lb_handle* h, double tol, int check, long long max_steps) {
    const size_t G = h->sweep_groups.size();
    const uint32_t key_sr = step_key(h, h->step + 0x5bd1e995ll);
    std::vector<double> key = {tol, (double)check, (double)max_steps, (double)key_sr};
    for (const SweepGroup& g : h->sweep_groups)
        for (int v : {g.begin, g.count, g.ny_min, g.ny_max, g.var, g.nt, g.cl}) key.push_back((double)v);
    if (!h->sweep_gexec || key != h->sweep_key || h->sweep_pin != h->popA) {
        if (h->sweep_gexec) {
            LB_CK(cudaGraphExecDestroy(h->sweep_gexec));
            h->sweep_gexec = nullptr;
        }
        if (!h->cap_stream) LB_CK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
        if (!h->fork_ev) LB_CK(cudaEventCreateWithFlags(&h->fork_ev, cudaEventDisableTiming));
        while (h->gstreams.size() < G) {
            cudaStream_t q = nullptr;
            cudaEvent_t ev = nullptr;
            LB_CK(cudaStreamCreateWithFlags(&q, cudaStreamNonBlocking));
            h->gstreams.push_back(q);
            LB_CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
            h->gevents.push_back(ev);
        }
        cudaStream_t cap = h->cap_stream;
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(e, "lb_run_until_steady: graph capture begin");
        e = cudaEventRecord(h->fork_ev, cap);
        for (size_t k = 0; k < G && e == cudaSuccess; ++k) {
            const SweepGroup& g = h->sweep_groups[k];
            e = cudaStreamWaitEvent(h->gstreams[k], h->fork_ev, 0);  // fork
            if (e != cudaSuccess) break;
            const cudaError_t el = sweep_launch_any(h, g, g.var, g.nt, g.cl, tol, check, max_steps, h->gstreams[k]);
            // join the forked stream whatever the launch did, so that no stream stays in capture
            e = cudaEventRecord(h->gevents[k], h->gstreams[k]);
            const cudaError_t ej = cudaStreamWaitEvent(cap, h->gevents[k], 0);
            if (e == cudaSuccess) e = ej;
            if (e == cudaSuccess) e = el;
        }
        cudaGraph_t graph = nullptr;
        const cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&h->sweep_gexec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            h->sweep_gexec = nullptr;
            return cuda_fail(e, "lb_run_until_steady: graph capture");
        }
        h->sweep_key = key;
        h->sweep_pin = h->popA;
    }
    LB_CK(cudaGraphLaunch(h->sweep_gexec, h->stream));
    return LB_OK;
}

}  // namespace

extern "C" {

const char* lb_last_error(void) { return g_err; }

lb_status lb_run_until_steady(lb_handle* h, double tol, long check_every, long max_steps, long long* steps_out,
                              double* residual_out) {
    NvtxRange range("lb_run_until_steady");
    if (!h || check_every < 2 || (check_every & 1) || max_steps < check_every || std::isnan(tol))
        return fail(LB_EINVAL, "lb_run_until_steady: need an even check_every >= 2 and max_steps >= check_every%s");
    if (h->smode != 0) return fail(LB_EINVAL, "lb_run_until_steady: the sweep kernel implements stress mode 0%s");
    if (h->gpbc || h->moving)
        return fail(LB_EINVAL, "lb_run_until_steady: the sweep kernel implements periodic x and bounce-back walls only%s");
    if (h->scheme != 0)
        return fail(LB_EINVAL, "lb_run_until_steady: the sweep kernel implements the paper's model only (step the comparison schemes and the relaxation-time extensions with lb_step)%s");
    if (h->prec == LB_PREC_F64S_F32M || h->prec == LB_PREC_F32S_F64M)
        return fail(LB_EINVAL, "lb_run_until_steady: diagnostic precision mixes are not supported%s");
    // Segments of growing length (64, 256, 1024, ... check intervals): after each one the
    // converged channels drop out and the classes that lost half of their channels are tuned
    // again, so the last, slowest channels run with the shape of lowest per-step latency.  A
    // channel's first check interval in a segment only saves its velocity.
    const long long ms = (long long)((max_steps + check_every - 1) / check_every) * check_every;
    std::vector<long long> total(h->n_ch, -3);   // -3: not run (unstable before)
    std::vector<double> res(h->n_ch, NAN);
    std::vector<char> active(h->n_ch, 1);
    std::vector<long long> seg_steps(h->n_ch);
    std::vector<double> seg_res(h->n_ch);
    long long done = 0, seg = 64LL * check_every;
    lb_status st = LB_OK;
    bool first = true;
    while (done < ms) {
        int n_active = 0;
        st = sweep_order(h, &n_active, &active);
        if (st != LB_OK) return st;
        if (n_active == 0) break;
        bool untuned = false;
        for (const SweepGroup& g : h->sweep_groups) untuned |= g.nt == 0;
        if (untuned) {
            st = sweep_tune(h, false);
            if (st != LB_OK) return st;
        }
        const long long L = std::min(seg, ms - done);
        std::vector<long long> init(h->n_ch, -3);
        LB_CK(cudaMemcpyAsync(h->sweep_steps_d, init.data(), sizeof(long long) * h->n_ch, cudaMemcpyHostToDevice, h->stream));
        st = sweep_run(h, tol, (int)check_every, L);
        if (st != LB_OK) return st;
        LB_CK(cudaMemcpyAsync(seg_steps.data(), h->sweep_steps_d, sizeof(long long) * h->n_ch, cudaMemcpyDeviceToHost, h->stream));
        LB_CK(cudaMemcpyAsync(seg_res.data(), h->sweep_res_d, sizeof(double) * h->n_ch, cudaMemcpyDeviceToHost, h->stream));
        LB_CK(cudaStreamSynchronize(h->stream));
        for (int c = 0; c < h->n_ch; ++c) {
            if (!active[c] || seg_steps[c] == -3) {
                if (first && active[c]) active[c] = 0;   // unstable before the sweep
                continue;
            }
            res[c] = seg_res[c];
            if (seg_steps[c] >= 0) {                     // converged in this segment
                total[c] = done + seg_steps[c];
                active[c] = 0;
            } else if (seg_steps[c] == -2) {             // became unstable
                total[c] = -2;
                active[c] = 0;
            } else {
                total[c] = -1;
            }
        }
        done += L;
        seg *= 4;
        first = false;
    }
    for (int c = 0; c < h->n_ch; ++c) {
        if (steps_out) steps_out[c] = total[c] == -3 ? -2 : total[c];
        if (residual_out) residual_out[c] = res[c];
    }
    h->uprev_state = -10;
    h->mon_state = -1;
    return LB_OK;
}

lb_status lb_sweep_tune(lb_handle* h) {
    NvtxRange range("lb_sweep_tune");
    if (!h) return fail(LB_EINVAL, "lb_sweep_tune: null handle%s");
    if (h->smode != 0) return fail(LB_EINVAL, "lb_sweep_tune: the sweep kernel implements stress mode 0%s");
    if (h->gpbc || h->moving)
        return fail(LB_EINVAL, "lb_sweep_tune: the sweep kernel implements periodic x and bounce-back walls only%s");
    int n_active = 0;
    lb_status st = sweep_order(h, &n_active);
    if (st != LB_OK || n_active == 0) return st;
    h->sweep_fixed = false;
    return sweep_tune(h, true);
}

int lb_sweep_variant(const lb_handle* h) {
    if (!h || h->sweep_groups.empty()) return -1;
    return h->sweep_groups[0].var;
}

int lb_sweep_groups(const lb_handle* h, int* variant, int* threads, int* cluster, int* channels, int max_groups) {
    if (!h) return -1;
    const int G = (int)h->sweep_groups.size();
    for (int k = 0; k < G && k < max_groups; ++k) {
        const SweepGroup& g = h->sweep_groups[k];
        if (variant) variant[k] = g.var;
        if (threads) threads[k] = g.nt;
        if (cluster) cluster[k] = g.cl;
        if (channels) channels[k] = g.count;
    }
    return G;
}

lb_status lb_sweep_set_config(lb_handle* h, int variant, int threads, int cluster) {
    if (!h || (variant != 0 && variant != 1) || (threads != 128 && threads != 256))
        return fail(LB_EINVAL, "lb_sweep_set_config: variant 0/1 and threads 128/256%s");
    if (h->smode != 0 || h->gpbc || h->moving) return fail(LB_EINVAL, "lb_sweep_set_config: not a sweep handle%s");
    int n_active = 0;
    lb_status st = sweep_order(h, &n_active);
    if (st != LB_OK) return st;
    for (const SweepGroup& g : h->sweep_groups)
        if (!sweep_config_fits(h, g, variant, threads, cluster) || sweep_capacity(h, g, variant, threads, cluster) < 1)
            return fail(LB_EINVAL, "lb_sweep_set_config: configuration does not fit these channels%s");
    for (SweepGroup& g : h->sweep_groups) {
        g.var = variant;
        g.nt = threads;
        g.cl = cluster;
        g.tune_ms = 0.0;
    }
    h->sweep_fixed = true;
    return LB_OK;
}

lb_status lb_sweep_config(lb_handle* h, int* threads, int* cluster, double* tune_ms) {
    if (!h) return fail(LB_EINVAL, "lb_sweep_config: null handle%s");
    const SweepGroup* g = h->sweep_groups.empty() ? nullptr : &h->sweep_groups[0];
    if (threads) *threads = g ? g->nt : 0;
    if (cluster) *cluster = g ? g->cl : 0;
    if (tune_ms) {
        double t = 0.0;
        for (const SweepGroup& q : h->sweep_groups) t += q.tune_ms;
        *tune_ms = t;
    }
    return LB_OK;
}

const char* lb_strerror(lb_status s) {
    switch (s) {
        case LB_OK: return "ok";
        case LB_EINVAL: return "invalid argument";
        case LB_ENOMEM: return "out of memory";
        case LB_ECUDA: return "CUDA error";
        case LB_EUNSTABLE: return "channel unstable";
        case LB_ETIMEOUT: return "device wait timed out";
        case LB_ESTATE: return "state not available";
    }
    return "unknown status";
}

lb_status lb_create(const lb_grid* grid, const lb_params* params, const lb_boundary* boundary, void* cuda_stream,
                    lb_handle** out) {
    if (!out) return fail(LB_EINVAL, "lb_create: out is null%s");
    *out = nullptr;
    lb_status st = validate(grid, params, boundary);
    if (st != LB_OK) return st;
    lb_handle* h = new (std::nothrow) lb_handle();
    if (!h) return fail(LB_ENOMEM, "lb_create: host allocation%s");
    auto bail = [&](lb_status s) { release(h); return s; };
    cudaGetDevice(&h->dev);
    h->stream = (cudaStream_t)cuda_stream;
    h->n_ch = grid->n_channels;
    h->nx = grid->nx;
    h->prec = grid->precision;
    h->smode = grid->stress_mode;
    h->flags = grid->flags;
    h->scheme = (grid->flags & LB_GRID_GENERALIZED_NEWTONIAN) ? 1 : ((grid->flags & LB_GRID_STRESS_DIVERGENCE) ? 2 : 0);
    if (grid->flags & LB_GRID_RELAXATION_MODEL) h->scheme = 3;
    h->tsize = with_types(h->prec, [](auto tt, auto tc) { LB_TYPES(tt, tc); (void)sizeof(C); return sizeof(T); });
    h->csize = with_types(h->prec, [](auto tt, auto tc) { LB_TYPES(tt, tc); (void)sizeof(T); return sizeof(C); });
    h->ny.assign(grid->ny, grid->ny + h->n_ch);
    h->params.assign(params, params + h->n_ch);
    h->beta_rho.assign(h->n_ch, 0.0);
    h->rho_ref.assign(h->n_ch, 1.0);
    h->tau_f.assign(h->n_ch, 0.0);
    h->P.resize(h->n_ch); h->base.resize(h->n_ch); h->node_off.resize(h->n_ch);
    long long acc = 0, nodes = 0;
    for (int c = 0; c < h->n_ch; ++c) {
        const long long n = (long long)h->nx * h->ny[c];
        h->P[c] = (n + 63) / 64 * 64;
        h->base[c] = acc;
        h->node_off[c] = nodes;
        acc += h->P[c];
        nodes += n;
    }
    h->planes = acc;
    h->nodes = nodes;
    h->gpbc = boundary->x_mode == LB_X_GPBC;
    h->moving = boundary->walls == LB_WALLS_COUETTE;
    h->u_wall.assign(h->n_ch, 0.0);
    h->row_off.resize(h->n_ch);
    for (int c = 0; c < h->n_ch; ++c) {
        h->row_off[c] = h->gny;
        h->gny += h->ny[c];
    }
    int n_sm = 0;
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, h->dev);
    plan_tiles(h, std::max(1, n_sm));

    auto dmalloc = [&](void** p, size_t bytes) -> cudaError_t { return cudaMalloc(p, bytes < 16 ? 16 : bytes); };
    cudaError_t e;
#define LB_ALLOC(ptr, bytes)                                                   \
    do {                                                                       \
        e = dmalloc((void**)&(ptr), (bytes));                                  \
        if (e != cudaSuccess) return bail(cuda_fail(e, "lb_create: cudaMalloc")); \
    } while (0)
    LB_ALLOC(h->popA, 9 * h->planes * h->tsize);
    LB_ALLOC(h->popB, 9 * h->planes * h->tsize);
    LB_ALLOC(h->drho, h->planes * h->csize);
    if (h->smode == 1) LB_ALLOC(h->sig3, 3 * h->planes * h->csize);
    if (h->scheme == 2) LB_ALLOC(h->snn, 3 * h->planes * h->csize);
    if (h->scheme == 3) LB_ALLOC(h->phi, h->planes * sizeof(double));  // FP64 in every precision
    if (h->flags & LB_GRID_STORE_SIGMA) LB_ALLOC(h->sig4, 4 * h->planes * h->csize);
    LB_ALLOC(h->uprev, 2 * h->planes * h->csize);
    LB_ALLOC(h->chan, h->n_ch * (h->csize == 8 ? sizeof(ChanParams<double>) : sizeof(ChanParams<float>)));
    LB_ALLOC(h->items_d, h->items.size() * sizeof(WorkItem));
    LB_ALLOC(h->item_begin_d, (h->n_ch + 1) * sizeof(int));
    LB_ALLOC(h->partials, 4 * h->items.size() * sizeof(double));
    LB_ALLOC(h->mon_d, 4 * h->n_ch * sizeof(double));
    LB_ALLOC(h->status_d, h->n_ch * sizeof(int));
    LB_ALLOC(h->base_d, h->n_ch * sizeof(long long));
    LB_ALLOC(h->P_d, h->n_ch * sizeof(long long));
    LB_ALLOC(h->node_off_d, h->n_ch * sizeof(long long));
    LB_ALLOC(h->ny_d, h->n_ch * sizeof(int));
    LB_ALLOC(h->gx_d, 2 * h->n_ch * sizeof(double));
    LB_ALLOC(h->done_count_d, sizeof(unsigned));
    if (h->gpbc) {
        for (int c = 0; c < h->n_ch; ++c) h->gpbc_max_ny = std::max(h->gpbc_max_ny, h->ny[c]);
        const size_t rb = ((size_t)h->gpbc_max_ny + 255) / 256;
        LB_ALLOC(h->gcol, (6 * (size_t)h->gny + 2 * h->n_ch) * h->csize);
        LB_ALLOC(h->gpart, 2 * h->n_ch * rb * sizeof(double));
        LB_ALLOC(h->gcount, 2 * h->n_ch * sizeof(unsigned));
    }
#undef LB_ALLOC
    e = cudaHostAlloc((void**)&h->status_h, h->n_ch * sizeof(int), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&h->status_hd, h->status_h, 0);
    if (e != cudaSuccess) return bail(cuda_fail(e, "lb_create: cudaHostAlloc (mapped)"));
    std::memset(h->status_h, 0, h->n_ch * sizeof(int));
    e = cudaHostAlloc((void**)&h->mon_h, 4 * (size_t)h->n_ch * sizeof(double), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&h->mon_hd, h->mon_h, 0);
    if (e != cudaSuccess) return bail(cuda_fail(e, "lb_create: cudaHostAlloc (mapped)"));
    e = cudaEventCreateWithFlags(&h->status_ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return bail(cuda_fail(e, "lb_create: cudaEventCreate"));

    // tables, in the order of the handle's stream (a cudaMemcpy from pageable memory may return before its data have
    // arrived, and a non-blocking stream does not wait for them); the stream is waited for below
    std::vector<double> gx(2 * h->n_ch, 0.0);
    std::vector<InitChan> ic(h->n_ch);
    for (int c = 0; c < h->n_ch; ++c) {
        gx[c] = h->params[c].g_x;
        const double half = 1.5 * h->params[c].g_x * (double)(h->nx + 1);
        ic[c] = InitChan{h->base[c], h->P[c], h->ny[c], h->gpbc ? 1 : 0, h->params[c].rho0, h->params[c].rho_pert_amp,
                         h->params[c].seed, h->params[c].rho0 + half, h->params[c].rho0 - half};
    }
    InitChan* ic_d = nullptr;
    e = cudaMalloc(&ic_d, sizeof(InitChan) * h->n_ch);
    if (e != cudaSuccess) return bail(cuda_fail(e, "lb_create: cudaMalloc"));
    bool ok = true;
    ok &= cudaMemcpyAsync(ic_d, ic.data(), sizeof(InitChan) * h->n_ch, cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    if (h->csize == 8) {
        auto v = make_chan<double>(h);
        ok &= cudaMemcpyAsync(h->chan, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
        ok &= cudaStreamSynchronize(h->stream) == cudaSuccess;  // (v goes)
    } else {
        auto v = make_chan<float>(h);
        ok &= cudaMemcpyAsync(h->chan, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
        ok &= cudaStreamSynchronize(h->stream) == cudaSuccess;  // (v goes)
    }
    ok &= cudaMemcpyAsync(h->items_d, h->items.data(), sizeof(WorkItem) * h->items.size(), cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(h->item_begin_d, h->item_begin.data(), sizeof(int) * (h->n_ch + 1), cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(h->base_d, h->base.data(), sizeof(long long) * h->n_ch, cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(h->P_d, h->P.data(), sizeof(long long) * h->n_ch, cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(h->node_off_d, h->node_off.data(), sizeof(long long) * h->n_ch, cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(h->ny_d, h->ny.data(), sizeof(int) * h->n_ch, cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(h->gx_d, gx.data(), sizeof(double) * 2 * h->n_ch, cudaMemcpyHostToDevice, h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(h->status_d, 0, sizeof(int) * h->n_ch, h->stream) == cudaSuccess;
    if (h->gcount) ok &= cudaMemsetAsync(h->gcount, 0, 2 * h->n_ch * sizeof(unsigned), h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(h->done_count_d, 0, sizeof(unsigned), h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(h->uprev, 0, 2 * h->planes * h->csize, h->stream) == cudaSuccess;
    ok &= cudaMemsetAsync(h->popB, 0, 9 * h->planes * h->tsize, h->stream) == cudaSuccess;
    if (h->sig4) ok &= cudaMemsetAsync(h->sig4, 0, 4 * h->planes * h->csize, h->stream) == cudaSuccess;
    if (h->phi) ok &= cudaMemsetAsync(h->phi, 0, h->planes * sizeof(double), h->stream) == cudaSuccess;
    if (!ok) { cudaFree(ic_d); return bail(cuda_fail(cudaGetLastError(), "lb_create: table upload")); }
    long long maxn = 0;
    for (int c = 0; c < h->n_ch; ++c) maxn = std::max(maxn, (long long)h->nx * h->ny[c]);
    dim3 g(grid_for(maxn), h->n_ch);
    with_types(h->prec, [&](auto tt, auto tc) {
        LB_TYPES(tt, tc);
        k_init<T, C><<<g, 256, 0, h->stream>>>((T*)h->popA, (C*)h->drho, (C*)h->sig3, ic_d, h->nx, h->smode);
        return 0;
    });
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    cudaFree(ic_d);
    if (e != cudaSuccess) return bail(cuda_fail(e, "lb_create: init kernel"));
    st = plan_march(h);
    if (st != LB_OK) return bail(st);
    plan_resident(h);
    *out = h;
    return LB_OK;
}

void lb_destroy(lb_handle* h) { release(h); }

lb_status lb_set_relaxation_model(lb_handle* h, int channel, double beta_rho, double rho_ref, double tau_f) {
    if (!h || channel < -1 || channel >= h->n_ch || !std::isfinite(beta_rho) || !std::isfinite(rho_ref) ||
        !(rho_ref > 0.0) || !std::isfinite(tau_f) || tau_f < 0.0)
        return fail(LB_EINVAL, "lb_set_relaxation_model: bad handle, channel or parameter%s");
    if (h->scheme != 3) return fail(LB_EINVAL, "lb_set_relaxation_model: the handle was created without LB_GRID_RELAXATION_MODEL%s");
    for (int c = 0; c < h->n_ch; ++c)
        if (channel < 0 || c == channel) {
            h->beta_rho[c] = beta_rho;
            h->rho_ref[c] = rho_ref;
            h->tau_f[c] = tau_f;
        }
    // the whole channel table again (its body forces and wall velocities are the host's current
    // ones), after the work already queued that reads the old table
    LB_CK(cudaStreamSynchronize(h->stream));
    if (h->csize == 8) {
        auto v = make_chan<double>(h);
        LB_CK(cudaMemcpyAsync(h->chan, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice, h->stream));
        LB_CK(cudaStreamSynchronize(h->stream));  // (v goes)
    } else {
        auto v = make_chan<float>(h);
        LB_CK(cudaMemcpyAsync(h->chan, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice, h->stream));
        LB_CK(cudaStreamSynchronize(h->stream));  // (v goes)
    }
    return LB_OK;
}

lb_status lb_set_wait_limit(lb_handle* h, double seconds) {
    if (!h || !(seconds >= 0.0) || seconds > 60.0) return fail(LB_EINVAL, "lb_set_wait_limit: need 0 <= seconds <= 60%s");
    h->wait_ns = (unsigned long long)(seconds * 1e9);
    return LB_OK;
}

long lb_step_count(const lb_handle* h) { return h ? h->step : -1; }
int lb_uses_row_march(const lb_handle* h) { return (h && h->march) ? 1 : 0; }

int lb_row_march_plan(int nx, int ny, int ctas_per_sm, int n_sm, int precision, int gpbc, int* items, int max_items) {
    if (nx <= 0 || nx % kMarchW != 0 || ny < 16 || ctas_per_sm < 1 || n_sm < 1 || max_items < 0 ||
        (precision != LB_PREC_F32 && precision != LB_PREC_BF16))
        return -LB_EINVAL;
    const std::vector<MarchItem> v = march_plan(nx, ny, ctas_per_sm, n_sm, march_model(precision, gpbc != 0, (long long)nx * ny));
    if (items) {
        if ((int)v.size() > max_items) return -LB_EINVAL;
        for (size_t i = 0; i < v.size(); ++i) {
            items[3 * i] = v[i].x0;
            items[3 * i + 1] = v[i].y0;
            items[3 * i + 2] = v[i].y1;
        }
    }
    return (int)v.size();
}
long lb_graph_replays(const lb_handle* h) { return h ? h->graph_replays : -1; }
size_t lb_num_nodes(const lb_handle* h) { return h ? (size_t)h->nodes : 0; }

lb_status lb_step(lb_handle* h, long n) {
    NvtxRange range("lb_step");
    if (!h || n < 0) return fail(LB_EINVAL, "lb_step: bad handle or n%s");
    lb_status st = poll_status(h, false);
    if (st != LB_OK) return st;
    if (h->any_timeout) return fail(LB_ETIMEOUT, "lb_step: a device-side wait timed out earlier%s");
    if (n == 0) return h->any_unstable ? LB_EUNSTABLE : LB_OK;
    st = with_types(h->prec, [&](auto tt, auto tc) { LB_TYPES(tt, tc); return run_steps<T, C>(h, n); });
    if (st != LB_OK) return st;
    if (!h->march && !h->status_pending) {
        st = request_status(h);
        if (st != LB_OK) return st;
    }
    return h->any_unstable ? LB_EUNSTABLE : LB_OK;
}

lb_status lb_get_fields(lb_handle* h, void* u, void* sigma, void* rho, int out_dtype, int on_device) {
    if (!h || (out_dtype != 0 && out_dtype != 1)) return fail(LB_EINVAL, "lb_get_fields: bad handle or dtype%s");
    if (!u && !sigma && !rho) return LB_OK;
    const long long N = h->nodes;
    const size_t osize = out_dtype == 0 ? 8 : 4;
    // buffers in device memory on 16-byte boundaries are written by the fields pass itself; anything else
    // (host memory, odd addresses) goes through the staging buffer
    auto direct = [h](const void* p) {
        if (!p) return true;
        cudaPointerAttributes at{};
        const bool ok = reinterpret_cast<uintptr_t>(p) % 16 == 0 && cudaPointerGetAttributes(&at, p) == cudaSuccess &&
                        ((at.type == cudaMemoryTypeDevice && at.device == h->dev) || at.type == cudaMemoryTypeManaged);
        (void)cudaGetLastError();
        return ok;
    };
    if (on_device && direct(u) && direct(sigma) && direct(rho)) return fields_pass(h, u, sigma, rho, out_dtype == 0);
    lb_status st = ensure_fields(h, osize);
    if (st != LB_OK) return st;
    const FieldParts f = field_parts(h, osize);
    st = fields_pass(h, u ? f.u : nullptr, sigma ? f.sigma : nullptr, rho ? f.rho : nullptr, out_dtype == 0);
    if (st != LB_OK) return st;
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    if (u) LB_CK(cudaMemcpyAsync(u, f.u, 2 * N * osize, kind, h->stream));
    if (sigma) LB_CK(cudaMemcpyAsync(sigma, f.sigma, 4 * N * osize, kind, h->stream));
    if (rho) LB_CK(cudaMemcpyAsync(rho, f.rho, N * osize, kind, h->stream));
    if (!on_device) LB_CK(cudaStreamSynchronize(h->stream));
    return LB_OK;
}

lb_status lb_monitor(lb_handle* h, double* out) {
    if (!h || !out) return fail(LB_EINVAL, "lb_monitor: null argument%s");
    if (h->mon_state < 0) return fail(LB_ESTATE, "lb_monitor: no monitor evaluated yet (run lb_step with n >= 2)%s");
    LB_CK(copy_out(h->mon_d, h->mon_hd, 4 * h->n_ch, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    std::memcpy(out, h->mon_h, 4 * h->n_ch * sizeof(double));
    return LB_OK;
}

lb_status lb_monitor_async(lb_handle* h, double* out) {
    if (!h || !out) return fail(LB_EINVAL, "lb_monitor_async: null argument%s");
    if (h->mon_state < 0) return fail(LB_ESTATE, "lb_monitor_async: no monitor evaluated yet (run lb_step with n >= 2)%s");
    // pinned host memory mapped into the device's address space (what cudaHostAlloc and torch's
    // pin_memory give under unified addressing) and this device's own memory: a one-block kernel
    // stores the values there; anything else (pageable host memory, managed memory, another device,
    // an address that is no multiple of 8) takes a stream-ordered copy
    cudaPointerAttributes at{};
    int dev = -1;
    const bool known = cudaPointerGetAttributes(&at, out) == cudaSuccess && at.devicePointer && cudaGetDevice(&dev) == cudaSuccess;
    if (known && (at.type == cudaMemoryTypeHost || (at.type == cudaMemoryTypeDevice && at.device == dev)) &&
        (uintptr_t)at.devicePointer % sizeof(double) == 0) {
        LB_CK(copy_out(h->mon_d, (double*)at.devicePointer, 4 * h->n_ch, h->stream));
    } else {
        (void)cudaGetLastError();
        LB_CK(cudaMemcpyAsync(out, h->mon_d, 4 * h->n_ch * sizeof(double), cudaMemcpyDefault, h->stream));
    }
    return LB_OK;
}

lb_status lb_set_monitor_mode(lb_handle* h, int mode) {
    if (!h || (mode != LB_MONITOR_RESIDUAL && mode != LB_MONITOR_FLUX_MAX))
        return fail(LB_EINVAL, "lb_set_monitor_mode: bad handle or mode%s");
    h->monitor_mode = mode;
    return LB_OK;
}

lb_status lb_residual(lb_handle* h, double* r) {
    if (!h || !r) return fail(LB_EINVAL, "lb_residual: null argument%s");
    if (h->mon_state >= 0 && !h->mon_resid)
        return fail(LB_ESTATE, "lb_residual: the last monitor evaluation had no residual (LB_MONITOR_FLUX_MAX)%s");
    std::vector<double> m(4 * (size_t)h->n_ch);
    lb_status st = lb_monitor(h, m.data());
    if (st != LB_OK) return st;
    for (int c = 0; c < h->n_ch; ++c) r[c] = m[4 * c];
    return LB_OK;
}

lb_status lb_set_body_force(lb_handle* h, int channel, double g_x) {
    if (!h || channel < -1 || channel >= h->n_ch || std::isnan(g_x) || std::isinf(g_x))
        return fail(LB_EINVAL, "lb_set_body_force: bad argument%s");
    if (channel >= 0) h->params[channel].g_x = g_x;
    else for (lb_params& p : h->params) p.g_x = g_x;
    return push_drive<false>(h, channel, g_x);
}

lb_status lb_set_wall_velocity(lb_handle* h, int channel, double u_wall) {
    if (!h || channel < -1 || channel >= h->n_ch || std::isnan(u_wall) || std::isinf(u_wall))
        return fail(LB_EINVAL, "lb_set_wall_velocity: bad argument%s");
    if (!h->moving) return fail(LB_EINVAL, "lb_set_wall_velocity: the handle has no moving wall%s");
    if (channel >= 0) h->u_wall[channel] = u_wall;
    else h->u_wall.assign(h->n_ch, u_wall);
    return push_drive<true>(h, channel, u_wall);
}

// The start state of every channel from device fields in node order (u [node][2], rho, drho or
// nullptr): equilibrium populations of (rho, u - f/(2 rho)), delta rho, zero carried stress.
static lb_status set_fields_dev(lb_handle* h, const double* su, const double* sr, const double* sd) {
    long long maxn = 0;
    for (int c = 0; c < h->n_ch; ++c) maxn = std::max(maxn, (long long)h->nx * h->ny[c]);
    dim3 g(grid_for(maxn), h->n_ch);
    with_types(h->prec, [&](auto tt, auto tc) {
        LB_TYPES(tt, tc);
        k_set_fields<T, C><<<g, 256, 0, h->stream>>>((T*)h->popA, (C*)h->drho, (C*)h->sig3, su, sr, sd,
                                                     h->base_d, h->P_d, h->node_off_d, h->ny_d, h->gx_d, h->nx, h->smode,
                                                     h->gpbc ? 1 : 0);
        return 0;
    });
    LB_CK(cudaGetLastError());
    if (h->phi) LB_CK(cudaMemsetAsync(h->phi, 0, h->planes * sizeof(double), h->stream));  // fluidity unset
    LB_CK(cudaStreamSynchronize(h->stream));
    h->uprev_state = -10;
    return LB_OK;
}

lb_status lb_set_fields(lb_handle* h, const double* u, const double* rho, const double* drho) {
    if (!h || !u || !rho) return fail(LB_EINVAL, "lb_set_fields: null argument%s");
    const long long N = h->nodes;
    lb_status st = ensure_hstage(h, (size_t)N * 4 * sizeof(double));
    if (st != LB_OK) return st;
    double* su = (double*)h->hstage;
    double* sr = su + 2 * N;
    double* sd = su + 3 * N;
    LB_CK(cudaMemcpyAsync(su, u, 2 * N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    LB_CK(cudaMemcpyAsync(sr, rho, N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    if (drho) LB_CK(cudaMemcpyAsync(sd, drho, N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    return set_fields_dev(h, su, sr, drho ? sd : nullptr);
}

// The warm start's tables and profile buffers, on the first call that gets them all: one that fails half-way (out of
// memory, in the middle of a stream capture) leaves the next to begin anew.
static lb_status ws_tables(lb_handle* h) {
    if (h->ws_ready) return LB_OK;
    for (void** q : {&h->ws_prm, &h->ws_row_off, &h->ws_rows, &h->ws_grid, &h->ws_scale}) free_dev(*q);
    LB_CK(cudaMalloc(&h->ws_prm, sizeof(WsChan) * h->n_ch));
    LB_CK(cudaMalloc(&h->ws_row_off, sizeof(int) * h->n_ch));
    LB_CK(cudaMalloc(&h->ws_rows, sizeof(double) * 3 * (size_t)h->gny));
    LB_CK(cudaMalloc(&h->ws_grid, sizeof(double) * 3 * 256 * (size_t)h->n_ch));
    LB_CK(cudaMalloc(&h->ws_scale, sizeof(double) * 3 * (size_t)h->n_ch));
    std::vector<WsChan> prm(h->n_ch);
    for (int c = 0; c < h->n_ch; ++c)
        prm[c] = WsChan{h->params[c].G_inf, h->params[c].tau0, h->params[c].theta, h->params[c].gamma_c};
    LB_CK(cudaMemcpyAsync(h->ws_row_off, h->row_off.data(), sizeof(int) * h->n_ch, cudaMemcpyHostToDevice, h->stream));
    LB_CK(cudaMemcpyAsync(h->ws_prm, prm.data(), sizeof(WsChan) * h->n_ch, cudaMemcpyHostToDevice, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));  // (prm goes)
    h->ws_ready = true;
    return LB_OK;
}

// Learned warm start: the closed-form steady profile of every channel (current parameters) on its
// rows and on the network grid, with the per-field scales.
static lb_status ws_closed_form(lb_handle* h) {
    lb_status st = ws_tables(h);
    if (st != LB_OK) return st;
    for (int c = 0; c < h->n_ch; ++c) {
        const lb_params& p = h->params[c];
        if (!(p.G_inf > 0.0) || !(p.tau0 > 0.0) || !(p.g_x > 0.0))
            return fail(LB_EINVAL, "lb_warmstart: every channel needs G_inf > 0, tau0 > 0 and g_x > 0 (the closed form)%s");
    }
    // (the body force, the only one that changes, is read from its stream-ordered device copy)
    LB_CK(launch_ws_closed_form(h->n_ch, (const WsChan*)h->ws_prm, h->gx_d, h->ny_d, (const int*)h->ws_row_off,
                                (double*)h->ws_rows, (double*)h->ws_grid, (double*)h->ws_scale, h->stream));
    return LB_OK;
}

lb_status lb_warmstart_apply(lb_handle* h, const float* pred, const float* t_mu, const float* t_sd) {
    if (!h || (!t_mu) != (!t_sd)) return fail(LB_EINVAL, "lb_warmstart_apply: null handle, or only one of t_mu, t_sd%s");
    lb_status st = ws_closed_form(h);
    if (st != LB_OK) return st;
    int n_sm = 0, max_ny = 0;
    LB_CK(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, h->dev));
    for (int v : h->ny) max_ny = std::max(max_ny, v);
    const cudaError_t e = with_types(h->prec, [&](auto tt, auto tc) {
        LB_TYPES(tt, tc);
        return launch_ws_start<T, C>(h->n_ch, max_ny, n_sm, pred, t_mu, t_sd, (const double*)h->ws_grid,
                                     (const double*)h->ws_scale, (const double*)h->ws_rows, h->gx_d, h->ny_d,
                                     (const int*)h->ws_row_off, h->base_d, h->P_d, h->nx, h->gpbc ? 1 : 0, (T*)h->popA,
                                     (C*)h->drho, h->smode == 1 ? (C*)h->sig3 : nullptr, h->stream);
    });
    if (e != cudaSuccess) return cuda_fail(e, "lb_warmstart_apply: start state");
    if (h->phi) LB_CK(cudaMemsetAsync(h->phi, 0, h->planes * sizeof(double), h->stream));  // fluidity unset
    LB_CK(cudaStreamSynchronize(h->stream));
    h->uprev_state = -10;
    return LB_OK;
}

lb_status lb_warmstart_targets(lb_handle* h, float* targets) {
    if (!h || !targets) return fail(LB_EINVAL, "lb_warmstart_targets: null argument%s");
    lb_status st = ws_closed_form(h);
    if (st != LB_OK) return st;
    st = ensure_fields(h, h->csize);
    if (st != LB_OK) return st;
    const FieldParts f = field_parts(h, h->csize);
    void *fu = f.u, *fs = f.sigma;
    st = fields_pass(h, fu, fs, nullptr, h->csize == 8);
    if (st != LB_OK) return st;
    if (h->csize == 8)
        LB_CK(launch_ws_targets<double>(h->n_ch, (const double*)fu, (const double*)fs, (const double*)h->ws_grid,
                                        (const double*)h->ws_scale, h->ny_d, h->node_off_d, h->nx, targets, h->stream));
    else
        LB_CK(launch_ws_targets<float>(h->n_ch, (const float*)fu, (const float*)fs, (const double*)h->ws_grid,
                                       (const double*)h->ws_scale, h->ny_d, h->node_off_d, h->nx, targets, h->stream));
    return LB_OK;
}

lb_status lb_set_populations(lb_handle* h, const double* n, const double* drho, const double* sig3) {
    if (!h || !n || !drho) return fail(LB_EINVAL, "lb_set_populations: null argument%s");
    const long long N = h->nodes;
    lb_status st = ensure_hstage(h, (size_t)N * 9 * sizeof(double));
    if (st != LB_OK) return st;
    long long maxn = 0;
    for (int c = 0; c < h->n_ch; ++c) maxn = std::max(maxn, (long long)h->nx * h->ny[c]);
    dim3 g(grid_for(maxn), h->n_ch);
    double* s = (double*)h->hstage;
    LB_CK(cudaMemcpyAsync(s, n, 9 * N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    with_types(h->prec, [&](auto tt, auto tc) {
        LB_TYPES(tt, tc);
        k_pop_from_f64<T, C><<<g, 256, 0, h->stream>>>((T*)h->popA, s, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
        return 0;
    });
    LB_CK(cudaGetLastError());
    LB_CK(cudaMemcpyAsync(s, drho, N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    if (h->csize == 8) k_planes_from_f64<double><<<g, 256, 0, h->stream>>>((double*)h->drho, s, 1, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
    else k_planes_from_f64<float><<<g, 256, 0, h->stream>>>((float*)h->drho, s, 1, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
    LB_CK(cudaGetLastError());
    if (h->smode == 1) {
        if (sig3) {
            LB_CK(cudaStreamSynchronize(h->stream));
            LB_CK(cudaMemcpyAsync(s, sig3, 3 * N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
            if (h->csize == 8) k_planes_from_f64<double><<<g, 256, 0, h->stream>>>((double*)h->sig3, s, 3, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
            else k_planes_from_f64<float><<<g, 256, 0, h->stream>>>((float*)h->sig3, s, 3, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
            LB_CK(cudaGetLastError());
        } else {
            LB_CK(cudaMemsetAsync(h->sig3, 0, 3 * h->planes * h->csize, h->stream));
        }
    }
    if (h->phi) LB_CK(cudaMemsetAsync(h->phi, 0, h->planes * sizeof(double), h->stream));  // fluidity unset
    LB_CK(cudaStreamSynchronize(h->stream));
    h->uprev_state = -10;
    return LB_OK;
}

lb_status lb_get_populations(lb_handle* h, double* n, double* drho, double* sig3) {
    if (!h || !n || !drho) return fail(LB_EINVAL, "lb_get_populations: null argument%s");
    const long long N = h->nodes;
    lb_status st = ensure_hstage(h, (size_t)N * 9 * sizeof(double));
    if (st != LB_OK) return st;
    long long maxn = 0;
    for (int c = 0; c < h->n_ch; ++c) maxn = std::max(maxn, (long long)h->nx * h->ny[c]);
    dim3 g(grid_for(maxn), h->n_ch);
    double* s = (double*)h->hstage;
    with_types(h->prec, [&](auto tt, auto tc) {
        LB_TYPES(tt, tc);
        k_pop_to_f64<T, C><<<g, 256, 0, h->stream>>>((const T*)h->popA, s, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
        return 0;
    });
    LB_CK(cudaGetLastError());
    LB_CK(cudaMemcpyAsync(n, s, 9 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    if (h->csize == 8) k_planes_to_f64<double><<<g, 256, 0, h->stream>>>((const double*)h->drho, s, 1, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
    else k_planes_to_f64<float><<<g, 256, 0, h->stream>>>((const float*)h->drho, s, 1, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
    LB_CK(cudaGetLastError());
    LB_CK(cudaMemcpyAsync(drho, s, N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    if (sig3 && h->smode == 1) {
        if (h->csize == 8) k_planes_to_f64<double><<<g, 256, 0, h->stream>>>((const double*)h->sig3, s, 3, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
        else k_planes_to_f64<float><<<g, 256, 0, h->stream>>>((const float*)h->sig3, s, 3, h->base_d, h->P_d, h->node_off_d, h->ny_d, h->nx);
        LB_CK(cudaGetLastError());
        LB_CK(cudaMemcpyAsync(sig3, s, 3 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
        LB_CK(cudaStreamSynchronize(h->stream));
    }
    return LB_OK;
}

namespace {
struct StateHeader {
    uint64_t magic, version;
    int64_t step, planes;
    int32_t n_ch, nx, prec, smode;
    uint64_t ny_hash;  // FNV-1a of the per-channel ny list: the image's channel split
    int32_t scheme, pad_;  // the planes an image carries depend on the scheme
};
constexpr uint64_t kMagic = 0x4d4c4e2d424c6772ull;
constexpr uint64_t kStateVersion = 2;

uint64_t ny_list_hash(const std::vector<int>& ny) {
    uint64_t x = 0xcbf29ce484222325ull;  // FNV-1a, 64-bit offset basis and prime
    for (int v : ny)
        for (int b = 0; b < 4; ++b) {
            x ^= (uint64_t)(((uint32_t)v >> (8 * b)) & 0xffu);
            x *= 0x100000001b3ull;
        }
    return x;
}
}  // namespace

size_t lb_state_bytes(const lb_handle* h) {
    if (!h) return 0;
    size_t b = sizeof(StateHeader) + 9 * h->planes * h->tsize + h->planes * h->csize;
    if (h->smode == 1) b += 3 * h->planes * h->csize;
    if (h->phi) b += h->planes * sizeof(double);
    return b;
}

lb_status lb_get_state(lb_handle* h, void* buf, size_t bytes) {
    if (!h || !buf || bytes < lb_state_bytes(h)) return fail(LB_EINVAL, "lb_get_state: bad buffer%s");
    StateHeader hd{kMagic, kStateVersion, h->step, h->planes, h->n_ch, h->nx, h->prec, h->smode, ny_list_hash(h->ny),
                   h->scheme, 0};
    char* p = (char*)buf;
    std::memcpy(p, &hd, sizeof hd);
    p += sizeof hd;
    LB_CK(cudaMemcpyAsync(p, h->popA, 9 * h->planes * h->tsize, cudaMemcpyDeviceToHost, h->stream));
    p += 9 * h->planes * h->tsize;
    LB_CK(cudaMemcpyAsync(p, h->drho, h->planes * h->csize, cudaMemcpyDeviceToHost, h->stream));
    p += h->planes * h->csize;
    if (h->smode == 1) LB_CK(cudaMemcpyAsync(p, h->sig3, 3 * h->planes * h->csize, cudaMemcpyDeviceToHost, h->stream));
    if (h->smode == 1) p += 3 * h->planes * h->csize;
    if (h->phi) LB_CK(cudaMemcpyAsync(p, h->phi, h->planes * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    return LB_OK;
}

lb_status lb_set_state(lb_handle* h, const void* buf, size_t bytes) {
    if (!h || !buf || bytes < lb_state_bytes(h)) return fail(LB_EINVAL, "lb_set_state: bad buffer%s");
    StateHeader hd;
    std::memcpy(&hd, buf, sizeof hd);
    if (hd.magic != kMagic || hd.version != kStateVersion)
        return fail(LB_EINVAL, "lb_set_state: not a state image of this library version%s");
    if (hd.planes != h->planes || hd.n_ch != h->n_ch || hd.nx != h->nx || hd.prec != h->prec || hd.scheme != h->scheme ||
        hd.smode != h->smode || hd.ny_hash != ny_list_hash(h->ny))
        return fail(LB_EINVAL, "lb_set_state: image does not match this handle's grid or channel split%s");
    const char* p = (const char*)buf + sizeof hd;
    LB_CK(cudaMemcpyAsync(h->popA, p, 9 * h->planes * h->tsize, cudaMemcpyHostToDevice, h->stream));
    p += 9 * h->planes * h->tsize;
    LB_CK(cudaMemcpyAsync(h->drho, p, h->planes * h->csize, cudaMemcpyHostToDevice, h->stream));
    p += h->planes * h->csize;
    if (h->smode == 1) LB_CK(cudaMemcpyAsync(h->sig3, p, 3 * h->planes * h->csize, cudaMemcpyHostToDevice, h->stream));
    if (h->smode == 1) p += 3 * h->planes * h->csize;
    if (h->phi) LB_CK(cudaMemcpyAsync(h->phi, p, h->planes * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    // a restored state starts healthy: the per-channel status word and the sticky flags are
    // cleared, so rolling back to a good image after an instability steps every channel again
    LB_CK(cudaMemsetAsync(h->status_d, 0, sizeof(int) * h->n_ch, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    h->status_pending = false;
    std::memset(h->status_h, 0, h->n_ch * sizeof(int));  // (the stream is idle: no kernel writes it now)
    h->any_unstable = h->any_timeout = false;
    h->step = hd.step;
    h->uprev_state = -10;
    h->mon_state = -1;
    return LB_OK;
}

lb_status lb_channel_status(lb_handle* h, int* status) {
    if (!h || !status) return fail(LB_EINVAL, "lb_channel_status: null argument%s");
    LB_CK(cudaMemcpyAsync(status, h->status_d, sizeof(int) * h->n_ch, cudaMemcpyDeviceToHost, h->stream));
    LB_CK(cudaStreamSynchronize(h->stream));
    for (int c = 0; c < h->n_ch; ++c) {
        if (status[c] & 1) h->any_unstable = true;
        if (status[c] & 2) h->any_timeout = true;
    }
    return LB_OK;
}

}  // extern "C"
