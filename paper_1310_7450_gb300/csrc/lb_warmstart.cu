// lb_warmstart.cu -- the learned warm start's profile arithmetic on the device (not in the paper):
// the closed-form steady channel profile of Sec. III B, the resampling between a channel's Ny rows
// and the network's 256-point grid, the encoding of steady LB profiles as training targets, and
// the decoding of network outputs into per-node start fields (u, rho = 1, delta rho).
//
// Grid: d = (y - y_c)/H at the centres of 256 equal cells, d_k = (k + 1/2)/256 * 2 - 1; rows:
// d_y = (y - (ny-1)/2)/(ny/2).  Resampling is linear interpolation with the end values held.
// Network target of field j on the grid: (profile - closed form) / scale_j, scale_j = max |closed
// form_j| (u_x, sigma_xy, N1).
#include <cuda_runtime.h>

#include <algorithm>

#include "lb_device.cuh"

namespace lbk {

constexpr int kWsGrid = 256;   // network grid points per field
constexpr int kWsPts = 4001;   // points of the trapezoid integration of the closed form
constexpr int kWsThreads = 256;

struct WsChan {
    double G, tau0, theta, gamma_c;  // G_inf, tau0, theta, gamma_c of the channel (the force is read where it is set)
};

__device__ inline double grid_d(int k) { return (k + 0.5) / kWsGrid * 2.0 - 1.0; }

// Square root of a positive normal number: the hardware's reciprocal square root, one Goldschmidt step and
// a final Newton correction by the residual (P. Markstein, IBM J. Res. Dev. 34, 1990): 7 FP64 operations,
// 0.500 units of the last place at most over 2^28 arguments of exponents within +-300.  Anything else (0 or subnormal, as
// at the wall of a fluid with a tiny critical strain) takes the library's.
__device__ __forceinline__ double ws_sqrt(double x) {
    if ((unsigned)__double2hiint(x) - 0x00100000u >= 0x7fe00000u) return sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double g = x * y, h = 0.5 * y;
    const double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    return fma(fma(-g, g, x), h, g);
}

// Padded index of point k of the integration in shared memory: a thread owns kWsPer consecutive points,
// and the padding spreads the threads' points over the banks.
constexpr int kWsPer = (kWsPts + kWsThreads - 1) / kWsThreads;
__device__ __forceinline__ int ws_pad(int k) { return k + k / kWsPer; }
constexpr int kWsPadded = kWsPts + kWsPts / kWsPer + 1;

// One CTA per channel: the closed-form steady profile (the quadratic for dv/dd of Sec. III B,
// v(1) = 0, integrated by the trapezoid rule on kWsPts points, u = (H/tau0) v) on the rows
// (rows[row_off + y][3] = u_x, sigma_xy, N1) and on the grid (grid[c][3][256]), and the scales.
//
// Bound by the part's FP64 rate (2 operations per SM and clock: 524e9/s measured).  Every point takes about
// 15 FP64 operations, 7 of them the square root: the point index is the abscissa (the step is folded
// into the coefficients), and the trapezoid sums come from one prefix sum of dv/dd, v_k = step
// (sum_{i<=k} dv_i - (dv_0 + dv_k)/2), formed where a row needs them.  The profile is even (u, N1) or odd
// (sigma_xy) about the middle, so rows and grid points are evaluated for one half.  512 channels of
// 32..1024 rows: 341 us with a division and a conversion per point, separate passes over the points
// and a serial sum of the threads' partial sums; 121 us now.
__global__ void __launch_bounds__(kWsThreads) k_ws_closed_form(const WsChan* __restrict__ prm,
                                                               const double* __restrict__ gx, const int* __restrict__ nys,
                                                               const int* __restrict__ row_off, double* __restrict__ rows,
                                                               double* __restrict__ grid, double* __restrict__ scale) {
    extern __shared__ double sh[];
    double* S = sh;                  // [kWsPadded] prefix sums of dv/dd
    double* dv = S + kWsPadded;      // [kWsPadded] dv/dd
    double* part = dv + kWsPadded;   // [kWsThreads / 32]
    const int c = blockIdx.x, t = threadIdx.x, ny = nys[c], lane = t & 31, w = t >> 5;
    const WsChan p = prm[c];
    const double H = ny / 2.0, wpH = gx[c] * H / p.G;
    const double step = 1.0 / (kWsPts - 1);
    // dv/dd = -a + b - sqrt((a - b)^2 + wpH d gamma_c / theta), a = wpH d / 2 (-wpH d at theta = 0),
    // at point kd
    const bool newt = p.theta == 0.0;
    const double ha = 0.5 * wpH * step;
    const double b = newt ? 0.0 : p.gamma_c * (1.0 + p.theta) / (2.0 * p.theta);
    const double q = newt ? 0.0 : wpH * step * p.gamma_c / p.theta;
    {
        const int k0 = t * kWsPer;
        double acc = 0.0, kd = (double)k0;
#pragma unroll 4
        for (int j = 0; j < kWsPer; ++j, kd += 1.0) {
            const int k = k0 + j;
            if (k < kWsPts) {
                const double x = fma(ha, kd, -b);
                const double r = newt ? -2.0 * x : -x - ws_sqrt(fma(x, x, q * kd));
                acc += r;
                dv[ws_pad(k)] = r;
                S[ws_pad(k)] = acc;
            }
        }
        // exclusive sums over the threads: within the warp, then over the warps
        double inc = acc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) part[w] = inc;
        __syncthreads();
        double off = inc - acc;
        for (int k = 0; k < w; ++k) off += part[k];
        for (int j = 0; j < kWsPer; ++j)
            if (k0 + j < kWsPts) S[ws_pad(k0 + j)] += off;
    }
    __syncthreads();
    const double dv0 = dv[0];
    auto integral = [&](int k) { return S[ws_pad(k)] - 0.5 * (dv0 + dv[ws_pad(k)]); };  // v_k / step
    const double vend = integral(kWsPts - 1);
    const double ku = H / p.tau0 * step, itau0 = 1.0 / p.tau0, igc = 1.0 / p.gamma_c, iH = 1.0 / H;
    const double tau = p.theta * p.tau0;
    double* crow = rows + 3LL * row_off[c];
    for (int y = t; y < (ny + 1) / 2; y += kWsThreads) {  // the half d <= 0, and its mirror image
        const double sd = fabs(y - (ny - 1) / 2.0) * iH * (kWsPts - 1);
        const int i = min((int)sd, kWsPts - 2);
        const double tt = sd - i;
        const double va = integral(i), da = dv[ws_pad(i)], db = dv[ws_pad(i + 1)];
        const double u = ku * (va + tt * (integral(i + 1) - va) - vend);
        const bool mid = 2 * y == ny - 1;
        const double gd = mid ? 0.0 : (da + tt * (db - da)) * itau0;
        const double tm = tau > 0.0 ? tau / (1.0 + tau * fabs(gd) * igc) : 0.0;
        const double sxy = p.G * tm * gd, n1 = 2.0 * p.G * gd * gd * tm * tm;
        double* r = crow + 3LL * y;
        r[0] = u;
        r[1] = -sxy;
        r[2] = n1;
        double* m = crow + 3LL * (ny - 1 - y);
        m[0] = u;
        m[1] = mid ? -sxy : sxy;
        m[2] = n1;
    }
    __syncthreads();  // (the block's global writes of the rows are visible to it after the barrier)
    double* gc = grid + 3LL * kWsGrid * c;
    double m[3] = {0.0, 0.0, 0.0};
    for (int k = t; k < kWsGrid / 2; k += kWsThreads) {
        // row coordinate of the grid point, end values held
        const double xr = fmin(fmax((grid_d(k) * H) + (ny - 1) / 2.0, 0.0), (double)(ny - 1));
        const int i = min((int)xr, ny - 2);
        const double tt = xr - i;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double fa = crow[3LL * i + j];
            const double g = fa + tt * (crow[3LL * i + 3 + j] - fa);
            gc[j * kWsGrid + k] = g;
            gc[j * kWsGrid + kWsGrid - 1 - k] = j == 1 ? -g : g;
            m[j] = fmax(m[j], fabs(g));
        }
    }
    for (int j = 0; j < 3; ++j) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[j] = fmax(m[j], __shfl_xor_sync(0xffffffffu, m[j], o));
        __syncthreads();
        if (lane == 0) part[w] = m[j];
        __syncthreads();
        if (t == 0) {
            double v = part[0];
            for (int k = 1; k < kWsThreads / 32; ++k) v = fmax(v, part[k]);
            scale[3 * c + j] = fmax(v, 1e-300);
        }
    }
}

// The start state of every channel from a network output (pred [c][768], standardised outputs;
// de-standardised with t_mu, t_sd when given) or, with pred == nullptr, from the closed form on the
// rows: u = (u_x(y), 0), rho = 1, delta rho = -(3/2) N1(y) (the trace of a simple-shear stress is N1;
// Eq. rhoplus), written as lb_set_fields writes it: the equilibrium of (rho, u - f/(2 rho)), no
// carried stress; no force and no delta rho with pressure-driven ends (gpbc).
// The state is the same in every column, so a row is decoded once (about 30 FP64 operations, the bound)
// and its nine populations are written nx times; the fields are not stored in between.  512 channels of
// 4 x 32..1024 nodes: decoding every node into FP64 fields and a second kernel over the nodes took
// 123 + 192 us, this 42 us.  Blocks share out the rows of channel blockIdx.y.
template <typename T, typename C>
__global__ void __launch_bounds__(kWsThreads) k_ws_start(const float* __restrict__ pred, const float* __restrict__ t_mu,
                                                         const float* __restrict__ t_sd, const double* __restrict__ grid,
                                                         const double* __restrict__ scale, const double* __restrict__ rows,
                                                         const double* __restrict__ gx, const int* __restrict__ nys,
                                                         const int* __restrict__ row_off, const long long* __restrict__ base,
                                                         const long long* __restrict__ P, int nx, int gpbc,
                                                         T* __restrict__ pop, C* __restrict__ drho, C* __restrict__ sig3) {
    __shared__ double prof[2][kWsGrid];      // decoded u_x and N1 on the grid
    __shared__ C val[kWsThreads][11];        // a chunk of rows: nine populations, delta rho (11: no bank conflicts)
    const int c = blockIdx.y, t = threadIdx.x, ny = nys[c];
    const int ya = (int)((long long)ny * blockIdx.x / gridDim.x), yb = (int)((long long)ny * (blockIdx.x + 1) / gridDim.x);
    if (pred) {
        for (int k = t; k < 2 * kWsGrid; k += kWsThreads) {
            const int jj = k / kWsGrid, j = jj == 0 ? 0 : 2;  // fields u_x and N1
            const int o = j * kWsGrid + k % kWsGrid;
            double y = (double)pred[(long long)c * 3 * kWsGrid + o];
            if (t_sd) y = y * (double)t_sd[o] + (double)t_mu[o];
            prof[jj][k % kWsGrid] = grid[3LL * kWsGrid * c + o] + scale[3 * c + j] * y;
        }
    }
    __syncthreads();
    const double iH = 2.0 / ny, hg = gpbc ? 0.0 : 0.5 * gx[c];
    T* pc = pop + 9 * base[c];
    C* dc = drho + base[c];
    const long long Pc = P[c];
    for (int y0 = ya; y0 < yb; y0 += kWsThreads) {
        const int y = y0 + t;
        if (y < yb) {
            double ux, n1;
            if (pred) {
                // grid coordinate of the row, end values held
                const double xg = fmin(fmax(((y - (ny - 1) / 2.0) * iH + 1.0) * (kWsGrid / 2) - 0.5, 0.0), kWsGrid - 1.0);
                const int i = min((int)xg, kWsGrid - 2);
                const double tt = xg - i;
                ux = prof[0][i] + tt * (prof[0][i + 1] - prof[0][i]);
                n1 = prof[1][i] + tt * (prof[1][i + 1] - prof[1][i]);
            } else {
                const double* r = rows + 3LL * (row_off[c] + y);
                ux = r[0];
                n1 = r[2];
            }
            ux -= hg;
            const double u2 = ux * ux, odd = 3.0 * ux, even = 3.0 * u2, none = -1.5 * u2;  // of 3 c.u + 4.5 (c.u)^2 - 1.5 u^2
#pragma unroll
            for (int i = 0; i < 9; ++i)
                val[t][i] = (C)(wgt<double>(i) * (cx(i) == 0 ? none : (cx(i) == 1 ? even + odd : even - odd)));
            val[t][9] = gpbc ? C(0) : (C)(-1.5 * n1);
        }
        __syncthreads();
        const int nr = min(kWsThreads, yb - y0);
        auto write = [&](int r, long long node) {
#pragma unroll
            for (int i = 0; i < 9; ++i) Store<T>::st(pc + i * Pc + node, val[r][i]);
            dc[node] = val[r][9];
            if (sig3)
                for (int j = 0; j < 3; ++j) sig3[3 * base[c] + j * Pc + node] = C(0);
        };
        if (nx <= 64) {
            for (int e = t; e < nr * nx; e += kWsThreads) write(e / nx, (long long)y0 * nx + e);
        } else {
            for (int r = 0; r < nr; ++r)
                for (int x = t; x < nx; x += kWsThreads) write(r, (long long)(y0 + r) * nx + x);
        }
        __syncthreads();
    }
}

// One CTA per channel: training targets from the fields of a state (u [node][2], sigma [node][4]
// as xx, yy, zz, xy; column x = 0 of each row): (profile - closed form)/scale on the grid, float.
template <typename F>
__global__ void __launch_bounds__(kWsThreads) k_ws_targets(const F* __restrict__ fu, const F* __restrict__ fs,
                                                           const double* __restrict__ grid, const double* __restrict__ scale,
                                                           const int* __restrict__ nys, const long long* __restrict__ node_off,
                                                           int nx, float* __restrict__ targets) {
    const int c = blockIdx.x, t = threadIdx.x, ny = nys[c];
    const double H = ny / 2.0, r0 = -(ny - 1) / 2.0 / H, rh = 1.0 / H;
    for (int k = t; k < kWsGrid; k += kWsThreads) {
        const double x = grid_d(k);
        // the row interval that holds x (end values held), then the three fields there
        double vals[3];
        if (x <= r0 || ny == 1) {
            const long long nd = node_off[c];
            vals[0] = (double)fu[2 * nd];
            vals[1] = (double)fs[4 * nd + 3];
            vals[2] = (double)fs[4 * nd] - (double)fs[4 * nd + 1];
        } else if (x >= r0 + (ny - 1) * rh) {
            const long long nd = node_off[c] + (long long)(ny - 1) * nx;
            vals[0] = (double)fu[2 * nd];
            vals[1] = (double)fs[4 * nd + 3];
            vals[2] = (double)fs[4 * nd] - (double)fs[4 * nd + 1];
        } else {
            int i = (int)floor((x - r0) / rh);
            if (i > ny - 2) i = ny - 2;
            const double tt = (x - (r0 + i * rh)) / rh;
            const long long na = node_off[c] + (long long)i * nx, nb = na + nx;
            const double ua = (double)fu[2 * na], ub = (double)fu[2 * nb];
            const double sa = (double)fs[4 * na + 3], sb = (double)fs[4 * nb + 3];
            const double qa = (double)fs[4 * na] - (double)fs[4 * na + 1], qb = (double)fs[4 * nb] - (double)fs[4 * nb + 1];
            vals[0] = ua + tt * (ub - ua);
            vals[1] = sa + tt * (sb - sa);
            vals[2] = qa + tt * (qb - qa);
        }
        for (int j = 0; j < 3; ++j) {
            const int o = j * kWsGrid + k;
            targets[(long long)c * 3 * kWsGrid + o] =
                (float)((vals[j] - grid[3LL * kWsGrid * c + o]) / scale[3 * c + j]);
        }
    }
}

cudaError_t launch_ws_closed_form(int n_ch, const WsChan* prm, const double* gx, const int* nys, const int* row_off,
                                  double* rows, double* grid, double* scale, cudaStream_t s) {
    const size_t smem = sizeof(double) * (2 * kWsPadded + kWsThreads / 32);
    cudaError_t e = cudaFuncSetAttribute(k_ws_closed_form, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_ws_closed_form<<<n_ch, kWsThreads, smem, s>>>(prm, gx, nys, row_off, rows, grid, scale);
    return cudaGetLastError();
}

template <typename T, typename C>
cudaError_t launch_ws_start(int n_ch, int max_ny, int n_sm, const float* pred, const float* t_mu, const float* t_sd,
                            const double* grid, const double* scale, const double* rows, const double* gx, const int* nys,
                            const int* row_off, const long long* base, const long long* P, int nx, int gpbc, T* pop, C* drho,
                            C* sig3, cudaStream_t s) {
    // blocks per channel: the chip filled about four times over, at least 32 rows each
    const int nb = std::max(1, std::min((max_ny + 31) / 32, (4 * n_sm + n_ch - 1) / n_ch));
    k_ws_start<T, C><<<dim3(nb, n_ch), kWsThreads, 0, s>>>(pred, t_mu, t_sd, grid, scale, rows, gx, nys, row_off, base, P, nx,
                                                           gpbc, pop, drho, sig3);
    return cudaGetLastError();
}
#define LB_WS_START(T, C)                                                                                                  \
    template cudaError_t launch_ws_start<T, C>(int, int, int, const float*, const float*, const float*, const double*,     \
                                               const double*, const double*, const double*, const int*, const int*,        \
                                               const long long*, const long long*, int, int, T*, C*, C*, cudaStream_t);
LB_WS_START(double, double)
LB_WS_START(float, float)
LB_WS_START(__nv_bfloat16, float)
LB_WS_START(double, float)
LB_WS_START(float, double)
#undef LB_WS_START

template <typename F>
cudaError_t launch_ws_targets(int n_ch, const F* fu, const F* fs, const double* grid, const double* scale, const int* nys,
                              const long long* node_off, int nx, float* targets, cudaStream_t s) {
    k_ws_targets<F><<<n_ch, kWsThreads, 0, s>>>(fu, fs, grid, scale, nys, node_off, nx, targets);
    return cudaGetLastError();
}
template cudaError_t launch_ws_targets<double>(int, const double*, const double*, const double*, const double*, const int*,
                                               const long long*, int, float*, cudaStream_t);
template cudaError_t launch_ws_targets<float>(int, const float*, const float*, const double*, const double*, const int*,
                                              const long long*, int, float*, cudaStream_t);

}  // namespace lbk
