// lb_step_resident.cuh -- many steps of one small channel in one launch, its state on chip.
//
// A step of a small channel is a chain of dependent instructions (about a microsecond) that a launch per step
// doubles or worse, and the tile kernel puts it on one or a few SMs.  Here one thread-block cluster owns the
// channel for a run of steps: CTA r keeps rows [ny r / CL, ny (r+1) / CL) of the populations in shared memory
// (two buffers, two halo rows on each side), one node per thread, delta rho and the carried stress in
// registers.  Per step:
//   1. pull-stream (Eq. lbupdate; bounce-back or Zou-He at the walls) from the current buffer; moments and
//      gradient velocity of the own nodes, and of one row on each side by further threads (same-time
//      gradients) -> shared velocity rows; barrier;
//   2. collision; the new populations go into the other buffer, those of the two rows next to a neighbour
//      also straight into its halo rows (distributed shared memory);
//   3. cluster barrier.
// The arithmetic is the tile kernel's, node by node: the same bits.  A node that fails the velocity guard raises
// a flag in every CTA, which all of them read after the cluster barrier: the channel stops there.
// us per step, launch per step in a graph -> here: FP32 4 x 64 3.2 -> 1.1, 20 x 400 4.2 -> 2.0, 4 x 1021 4.1 -> 1.6;
// FP64 4 x 64 10.7 -> 6.9, 4 x 256 10.9 -> 7.0.
// FP64: a warp's FP64 instruction takes 64 clocks on its quarter of the SM, however few lanes are active and whether
// or not the next one depends on it, and four warps run side by side; so up to 128 threads per CTA (one warp per
// quarter) a step costs the instructions of one node, and beyond that the tile kernel on all SMs is faster.
#pragma once

#include <cooperative_groups.h>

#include "lb_step_tile.cuh"

namespace lbk {

namespace cg = cooperative_groups;

constexpr int kResHalo = 2;  // halo rows of populations on each side

// Largest number of rows of a CTA, threads that work, dynamic shared memory of the kernel.
__host__ __device__ constexpr int resident_rows(int ny, int cl) { return (ny + cl - 1) / cl; }
constexpr int resident_threads(int ny, int nx, int cl) { return resident_rows(ny, cl) * nx + (cl > 1 ? 2 * nx : 0); }
template <typename T, typename C>
constexpr size_t resident_smem(int ny, int nx, int cl) {
    const size_t rows = resident_rows(ny, cl);
    return (2 * 9 * (rows + 2 * kResHalo) * nx * sizeof(T) + 15) / 16 * 16 + (rows + 2) * nx * 2 * sizeof(C);
}

template <typename T, typename C, int SMODE, int NT>
__global__ void __launch_bounds__(NT) k_step_resident(const StepArgs<T, C> a, T* pop, long long steps) {
    cg::cluster_group cluster = cg::this_cluster();
    const int CL = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    if (a.status[0] != 0) return;  // retired channel (uniform for the cluster)
    const ChanParams<C> P = a.chan[0];
    const int nx = a.nx, ny = P.ny, t = threadIdx.x;
    const int y0 = (int)((long long)ny * rank / CL), y1 = (int)((long long)ny * (rank + 1) / CL), n = y1 - y0;
    const int rmax = resident_rows(ny, CL);
    const int PS = (rmax + 2 * kResHalo) * nx;   // plane stride (the same in every CTA)

    extern __shared__ __align__(16) unsigned char smem[];
    T* buf = reinterpret_cast<T*>(smem);         // [2][9][rows][nx]; local row 0 is global row y0 - 2
    using V2 = typename Vec2<C>::type;
    V2* uv = reinterpret_cast<V2*>(smem + ((size_t)2 * 9 * PS * sizeof(T) + 15) / 16 * 16);  // [n + 2][nx], row 0: y0 - 1
    // raised in every CTA by a node that fails the velocity guard: one flag for even and one for odd steps, so that
    // a CTA already in the next step cannot raise the one that others have yet to read
    __shared__ int s_stop[2];
    if (t < 2) s_stop[t] = 0;

    T* gpop = pop + 9 * P.base;
    {   // own rows and the halo rows that exist
        const int ya = max(y0 - kResHalo, 0), cnt = (min(y1 + kResHalo, ny) - ya) * nx;
        for (int i = 0; i < 9; ++i)
            for (int e = t; e < cnt; e += blockDim.x)
                buf[i * PS + (ya - y0 + kResHalo) * nx + e] = gpop[(long long)i * P.P + (long long)ya * nx + e];
    }
    // this thread's node: an own node, or one of a neighbouring row (velocity only)
    const bool own = t < n * nx;
    const int h = t - n * nx;
    const int x = own ? t % nx : (h >= 0 ? h % nx : 0);
    const int y = own ? y0 + t / nx : (h < nx ? y0 - 1 : y1);
    const bool node = own || (h >= 0 && h < 2 * nx && y >= 0 && y < ny);
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    const int lr = (y - y0 + kResHalo) * nx;     // local row
    int off[9];                                  // where each population is pulled from
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ys = y - cy(i);
        off[i] = ys < 0 || ys >= ny ? opp(i) * PS + lr + x
                                    : i * PS + lr - cy(i) * nx + (cx(i) == 0 ? x : (cx(i) == 1 ? xm : xp));
        if (!node) off[i] = 0;
    }
    const int ur = (y - y0 + 1) * nx;            // velocity row
    const long long pn = (long long)y * nx + x;
    C drho = C(0), so_xx = C(0), so_xy = C(0), so_yy = C(0);
    if (own) {
        drho = a.drho[P.base + pn];
        if (SMODE == 1) {
            const C* s3 = a.sig3 + 3 * P.base + pn;
            so_xx = s3[0];
            so_xy = s3[P.P];
            so_yy = s3[2 * P.P];
        }
    }
    // halo rows of the neighbours that this node's new populations also belong to
    T* down = nullptr;
    T* up = nullptr;
    if (own && rank > 0 && y - y0 < kResHalo) {
        const int nb = y0 - (int)((long long)ny * (rank - 1) / CL);  // its rows
        down = cluster.map_shared_rank(buf, rank - 1) + (kResHalo + nb + (y - y0)) * nx + x;
    }
    if (own && rank < CL - 1 && y1 - y <= kResHalo)
        up = cluster.map_shared_rank(buf, rank + 1) + (kResHalo - (y1 - y)) * nx + x;
    const bool moving_row = P.moving && y == ny - 1;
    const bool store_sigma = (a.flags & F_STORE_SIGMA) != 0;
    C* s4 = a.sig4 + 4 * P.base + pn;
    cluster.sync();

    int cur = 0, stop = 0;  // element offset of the current buffer
    for (long long s = 0; s < steps && !stop; ++s) {
        const int nxt = cur == 0 ? 9 * PS : 0;
        C d[9], dR = C(0), jx = C(0), jy = C(0);
        if (node) {
            C ux, uy;
#pragma unroll
            for (int i = 0; i < 9; ++i) d[i] = (C)Store<T>::cvt(buf[cur + off[i]]);
            if (moving_row) zou_he_top<C>(d, P.u_wall);
            gradient_velocity<C>(d, P.gx, dR, jx, jy, ux, uy);
            V2 v;
            v.x = ux;
            v.y = uy;
            uv[ur + x] = v;
        }
        __syncthreads();
        if (own) {
            const V2 ue = uv[ur + xp], uw = uv[ur + xm];
            C B, Y;
            if (y == 0) {
                const V2 u0 = uv[ur + x], u1 = uv[ur + nx + x], u2 = uv[ur + 2 * nx + x];
                B = first_row_difference<C>(u0.x, u1.x, u2.x);
                Y = first_row_difference<C>(u0.y, u1.y, u2.y);
            } else if (y == ny - 1) {
                const V2 u0 = uv[ur + x], u1 = uv[ur - nx + x], u2 = uv[ur - 2 * nx + x];
                B = last_row_difference<C>(u0.x, u1.x, u2.x);
                Y = last_row_difference<C>(u0.y, u1.y, u2.y);
            } else {
                const V2 un = uv[ur + nx + x], us = uv[ur - nx + x];
                B = un.x - us.x;
                Y = un.y - us.y;
            }
            const NodeState<C> st = constitutive2<C, SMODE>(P, ue.x - uw.x, B, ue.y - uw.y, Y, dR, jx, jy, drho, so_xx, so_xy, so_yy);
            const C rho_h = C(1) + st.dReq - st.drho;
            if (!velocity_ok<C>(jx, jy, rho_h, a.guard)) {
                atomicOr(a.status, 1);
                for (int r = 0; r < CL; ++r) *cluster.map_shared_rank(&s_stop[s & 1], r) = 1;
            }
            C nw[9];
            collide_node<C>(P, st, d, dR, jx, jy, nw);
            drho = st.drho;
            if (SMODE == 1) {
                so_xx = st.sxx;
                so_xy = st.sxy;
                so_yy = st.syy;
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                T v;
                Store<T>::st(&v, nw[i]);
                buf[nxt + i * PS + lr + x] = v;
                if (down) down[nxt + i * PS] = v;
                if (up) up[nxt + i * PS] = v;
            }
            if (store_sigma) {  // (the zz plane holds 0 from lb_create on)
                s4[0] = st.sxx;
                s4[P.P] = st.syy;
                s4[3 * P.P] = st.sxy;
            }
        }
        cluster.sync();
        cur = nxt;
        stop = s_stop[s & 1];
    }
    // the state after the last step, back into the buffer it came from; a stopped channel's also into the other
    // one: the host goes on swapping the two for steps that do nothing
    if (own) {
#pragma unroll
        for (int i = 0; i < 9; ++i) gpop[(long long)i * P.P + pn] = buf[cur + i * PS + lr + x];
        if (stop) {
            T* other = a.pout + 9 * P.base;
#pragma unroll
            for (int i = 0; i < 9; ++i) other[(long long)i * P.P + pn] = buf[cur + i * PS + lr + x];
        }
        a.drho[P.base + pn] = drho;
        if (SMODE == 1) {
            C* s3 = a.sig3 + 3 * P.base + pn;
            s3[0] = so_xx;
            s3[P.P] = so_xy;
            s3[2 * P.P] = so_yy;
        }
    }
}

inline void resident_launch_config(int cl, int threads, size_t smem, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(cl);
    cfg->blockDim = dim3((threads + 31) / 32 * 32);
    cfg->dynamicSmemBytes = smem;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = cl;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
}

// Clusters of this shape the device holds at once (0: it cannot be launched), and the launch (after that question, which
// sets the kernel's limits).
template <typename T, typename C, int SMODE, int NT>
cudaError_t resident_capacity(int cl, int threads, size_t smem, int* clusters) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    auto k = k_step_resident<T, C, SMODE, NT>;
    resident_launch_config(cl, threads, smem, &cfg, attr);
    const cudaError_t e = allow_shared_memory(k);
    return e == cudaSuccess ? cudaOccupancyMaxActiveClusters(clusters, k, &cfg) : e;
}
template <typename T, typename C, int SMODE, int NT>
cudaError_t launch_step_resident(const StepArgs<T, C>& a, T* pop, long long steps, int cl, int threads, size_t smem,
                                 cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    resident_launch_config(cl, threads, smem, &cfg, attr);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, k_step_resident<T, C, SMODE, NT>, a, pop, steps);
}

// X(T, C, SMODE, NT): the kernel's instantiations; NT bounds the threads (and so the registers) of a CTA.
#define LB_RESIDENT_VARIANTS(X)                                                                     \
    X(double, double, 0, 128) X(double, double, 1, 128) X(float, float, 0, 128) X(float, float, 1, 128) \
    X(float, float, 0, 320) X(float, float, 1, 320) X(float, float, 0, 640) X(float, float, 1, 640)     \
    X(__nv_bfloat16, float, 0, 128) X(__nv_bfloat16, float, 1, 128) X(__nv_bfloat16, float, 0, 320)     \
    X(__nv_bfloat16, float, 1, 320) X(__nv_bfloat16, float, 0, 640) X(__nv_bfloat16, float, 1, 640)
#define LB_RESIDENT(PREFIX, T, C, SMODE, NT)                                                                          \
    PREFIX template cudaError_t resident_capacity<T, C, SMODE, NT>(int, int, size_t, int*);                           \
    PREFIX template cudaError_t launch_step_resident<T, C, SMODE, NT>(const StepArgs<T, C>&, T*, long long, int, int, \
                                                                      size_t, cudaStream_t);

}  // namespace lbk
