// lb_sweep_pair.cuh -- the shared-memory resident sweep in FP32 arithmetic, two nodes at a time.
//
// The contract of k_sweep_smem (lb_sweep_smem.cuh): one thread-block cluster per channel runs that channel's time
// loop with the populations in shared memory (two buffers), delta rho and the saved velocity in registers,
// until the residual over the check interval, an instability or max_steps ends it.  What differs:
//   - a thread's nodes go through the arithmetic in pairs, as packed FP32 (lb_pair.cuh): the sweep is bound by
//     instruction issue, and a pair takes one issue slot per operation;
//   - where a population comes from is a node's own offset plus a constant per direction, with the wall rows'
//     three exceptions patched in afterwards, instead of a range check and an index per direction;
//   - a node next to another CTA's rows writes its new populations into that CTA's halo rows as it
//     collides (distributed shared memory), so nothing is copied after the cluster barrier; two halo rows of
//     populations and one of velocities on each side.
// The host requires ny / CL >= 3.  Same bits as k_sweep_smem and lb_step.
// ms for 2000 steps of 4-column channels of 32..1024 rows, node by node -> here: 128 channels 16.7 -> 11.8, 512
// channels 45.0 -> 36.4, one of 1000 rows 4.07 -> 3.29.  Four blocks of 128 threads per SM (128 registers):
// three (168) take 16.5 / 42.7 / 3.14, five (96) 11.7 / 35.7 / 3.67.
#pragma once

#include <cooperative_groups.h>

#include "lb_pair.cuh"
#include "lb_sweep.cuh"

namespace lbk {

constexpr int kPairHalo = 2;  // halo rows of populations on each side

// Dynamic shared memory for CTAs of at most `rows` rows.
template <typename T>
constexpr size_t sweep_pair_smem(int rows, int nx) {
    return ((size_t)2 * 9 * (rows + 2 * kPairHalo) * nx * sizeof(T) + 15) / 16 * 16 + (size_t)(rows + 2) * nx * sizeof(float2);
}

// NT threads per CTA, NP pairs of nodes per thread (rows * nx <= 2 NT NP).  NX > 0: the width as a constant.
template <typename T, int NT, int NP, int NX = 0>
__global__ void __launch_bounds__(NT, 512 / NT) k_sweep_pair(const SweepArgs<T, float> a) {
    using C = float;
    cg::cluster_group cluster = cg::this_cluster();
    const int CL = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int ch = a.order[blockIdx.x / CL];
    const ChanParams<C> P = a.chan[ch];
    const PairConst q = pair_const(P);
    const int nx = NX > 0 ? NX : a.nx, ny = P.ny, t = threadIdx.x;
    const int y0 = (int)((long long)ny * rank / CL), y1 = (int)((long long)ny * (rank + 1) / CL);
    const int n_own = (y1 - y0) * nx;
    const int PS = ((ny + CL - 1) / CL + 2 * kPairHalo) * nx;  // plane stride, the same in every CTA of the channel

    extern __shared__ __align__(16) unsigned char smem[];
    T* buf = reinterpret_cast<T*>(smem);                       // [2][9][rows][nx], local row 0 is row y0 - 2
    float2* uv = reinterpret_cast<float2*>(smem + ((size_t)2 * 9 * PS * sizeof(T) + 15) / 16 * 16);  // row 0: y0 - 1
    __shared__ double part[2];
    __shared__ int done;

    T* gpop = a.popA + 9 * P.base;                             // the state at launch, and at exit
    C* gdr = a.drho + P.base;
    if (t == 0) done = 0;
    {   // own rows and the halo rows that exist
        const int ya = max(y0 - kPairHalo, 0), cnt = (min(y1 + kPairHalo, ny) - ya) * nx;
        for (int i = 0; i < 9; ++i)
            for (int e = t; e < cnt; e += NT)
                buf[i * PS + (ya - y0 + kPairHalo) * nx + e] = gpop[(long long)i * P.P + (long long)ya * nx + e];
    }
    // own nodes e = y * nx + x of rows y0.., pair p of this thread: nodes t + 2p NT and t + (2p + 1) NT (a missing
    // second node repeats the first and stores nothing)
    auto own_a = [&](int p) { return t + 2 * p * NT < n_own; };
    auto own_b = [&](int p) { return t + (2 * p + 1) * NT < n_own; };
    auto node_a = [&](int p) { return t + 2 * p * NT; };
    auto node_b = [&](int p) { return own_b(p) ? t + (2 * p + 1) * NT : t + 2 * p * NT; };
    auto west = [&](int e) { return e % nx == 0 ? nx - 1 : -1; };
    auto east = [&](int e) { return e % nx == nx - 1 ? 1 - nx : 1; };
    P2 drv[NP], upx[NP], upy[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        drv[p] = upx[p] = upy[p] = p2(0.f);
        if (own_a(p)) drv[p] = p2(gdr[(long long)y0 * nx + node_a(p)], gdr[(long long)y0 * nx + node_b(p)]);
    }
    cluster.sync();

    // pulled populations of the node with own index e (-nx .. n_own + nx - 1: a neighbouring row too)
    auto pull = [&](const T* cur, int e, C (&d)[9]) {
        const T* s = cur + kPairHalo * nx + e;
        const int w = west(e + nx), o = east(e + nx);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int c = cx(i) == 0 ? 0 : (cx(i) == 1 ? w : o);
            d[i] = (C)Store<T>::cvt(s[i * PS - cy(i) * nx + c]);
        }
        const int y = e + y0 * nx;  // bounce-back at the walls
        if (y < nx) {
            d[2] = (C)Store<T>::cvt(s[4 * PS]);
            d[5] = (C)Store<T>::cvt(s[7 * PS]);
            d[6] = (C)Store<T>::cvt(s[8 * PS]);
        }
        if (y >= (ny - 1) * nx) {
            d[4] = (C)Store<T>::cvt(s[2 * PS]);
            d[7] = (C)Store<T>::cvt(s[5 * PS]);
            d[8] = (C)Store<T>::cvt(s[6 * PS]);
        }
    };
    // the neighbouring rows' velocities: one node per thread, on the threads with the fewest own nodes
    const int spare = t - n_own % NT, h = spare >= 0 ? spare : spare + NT;
    const int below = y0 > 0 ? nx : 0, above = y1 < ny ? nx : 0;
    const bool pushes = CL > 1;

    long long s = 0;
    int dec = 0;
    for (; s < a.max_steps; ++s) {
        const T* cur = buf + ((s & 1) ? 9 * PS : 0);
        T* nxt = buf + ((s & 1) ? 0 : 9 * PS);
        const bool save = ((s + 1) % a.check) == 0;
        const bool resid = save && (s + 1 >= 2 * (long long)a.check);

        // 1. own nodes (kept in registers) and the neighbouring rows -> gradient velocity in shared memory
        P2 d[NP][9], dR[NP], jx[NP], jy[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (own_a(p)) {
                C da[9], db[9];
                pull(cur, node_a(p), da);
                pull(cur, node_b(p), db);
#pragma unroll
                for (int i = 0; i < 9; ++i) d[p][i] = p2(da[i], db[i]);
                P2 ux, uy;
                gradient_velocity(d[p], q.hgx, dR[p], jx[p], jy[p], ux, uy);
                uv[nx + node_a(p)] = make_float2(lo(ux), lo(uy));
                if (own_b(p)) uv[nx + node_b(p)] = make_float2(hi(ux), hi(uy));
            }
        }
        for (int k = h; k < below + above; k += NT) {
            const int e = k < below ? k - nx : n_own + (k - below);
            C dh[9], hR, hx, hy, ux, uy;
            pull(cur, e, dh);
            gradient_velocity<C>(dh, P.gx, hR, hx, hy, ux, uy);
            uv[nx + e] = make_float2(ux, uy);
        }
        __syncthreads();

        // 2. collide the own nodes into the other buffer
        P2 r0 = p2(0.f), r1 = p2(0.f);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (own_a(p)) {
                const int ea = node_a(p), eb = node_b(p);
                const float2* ua = uv + nx + ea;
                const float2* ub = uv + nx + eb;
                const float2 eA = ua[east(ea)], wA = ua[west(ea)], eB = ub[east(eb)], wB = ub[west(eb)];
                float2 nA = ua[nx], sA = ua[-nx], nB = ub[nx], sB = ub[-nx];
                const P2 Kx = p2(__fsub_rn(eA.x, wA.x), __fsub_rn(eB.x, wB.x));
                const P2 Kc = p2(__fsub_rn(eA.y, wA.y), __fsub_rn(eB.y, wB.y));
                float bA = __fsub_rn(nA.x, sA.x), yA = __fsub_rn(nA.y, sA.y);
                float bB = __fsub_rn(nB.x, sB.x), yB = __fsub_rn(nB.y, sB.y);
                auto wall = [&](int e, const float2* u, const float2& un, const float2& us, float& b, float& yy) {
                    if (e + y0 * nx < nx) {
                        const float2 u0 = u[0], u2 = u[2 * nx];
                        b = lo(wall_difference_first(p2(u0.x), p2(un.x), p2(u2.x)));
                        yy = lo(wall_difference_first(p2(u0.y), p2(un.y), p2(u2.y)));
                    }
                    if (e + y0 * nx >= (ny - 1) * nx) {
                        const float2 u0 = u[0], u2 = u[-2 * nx];
                        b = lo(wall_difference_last(p2(u0.x), p2(us.x), p2(u2.x)));
                        yy = lo(wall_difference_last(p2(u0.y), p2(us.y), p2(u2.y)));
                    }
                };
                wall(ea, ua, nA, sA, bA, yA);
                wall(eb, ub, nB, sB, bB, yB);
                const PairState st = constitutive<0, false, false>(q, Kx, p2(bA, bB), Kc, p2(yA, yB), dR[p], jx[p], jy[p], drv[p],
                                                                   p2(0.f), p2(0.f), p2(0.f), p2(0.f));
                const P2 rho_h = sub(add(p2(1.f), st.dReq), st.drho);
                {
                    const P2 j2 = fma(jy[p], jy[p], mul(jx[p], jx[p])), g2 = mul(mul(p2(0.3f * 0.3f), rho_h), rho_h);
                    if (!(lo(j2) <= lo(g2)) | !(hi(j2) <= hi(g2))) atomicOr(a.status + ch, 1);
                }
                P2 D[9];
                collide<false>(q, st, d[p], D, q.om, q.nom, q.k2);
                drv[p] = st.drho;
                auto put = [&](int e, const C (&n)[9]) {
                    T* o = nxt + kPairHalo * nx + e;
                    const uint32_t key = a.sr ? mix32(a.sr_key ^ (uint32_t)(s * 0x9E3779B9ull) ^ (uint32_t)(ch * 0x85EBCA6Bu)) : 0u;
                    store_node<T, C>(o, PS, n, a.sr, key, (uint32_t)(e + y0 * nx));
                    if (pushes) {
                        if (rank > 0 && e < kPairHalo * nx) {
                            const int nb = y0 - (int)((long long)ny * (rank - 1) / CL);  // the neighbour's rows
                            T* r = cluster.map_shared_rank(nxt, rank - 1) + (kPairHalo + nb) * nx + e;
                            for (int i = 0; i < 9; ++i) r[i * PS] = o[i * PS];
                        }
                        if (rank < CL - 1 && e >= n_own - kPairHalo * nx) {
                            T* r = cluster.map_shared_rank(nxt, rank + 1) + kPairHalo * nx + (e - n_own);
                            for (int i = 0; i < 9; ++i) r[i * PS] = o[i * PS];
                        }
                    }
                };
                C nA9[9], nB9[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const P2 v = add(d[p][i], D[i]);
                    nA9[i] = lo(v);
                    nB9[i] = hi(v);
                }
                put(ea, nA9);
                if (own_b(p)) put(eb, nB9);
                if (save) {
                    const P2 ih = rcp(rho_h);
                    const P2 urx = mul(jx[p], ih), ury = mul(jy[p], ih);
                    if (resid) {
                        const P2 dx_ = sub(urx, upx[p]), dy_ = sub(ury, upy[p]);
                        const P2 du2 = fma(dy_, dy_, mul(dx_, dx_)), u2 = fma(ury, ury, mul(urx, urx));
                        r0 = add(r0, p2(lo(du2), own_b(p) ? hi(du2) : 0.f));
                        r1 = add(r1, p2(lo(u2), own_b(p) ? hi(u2) : 0.f));
                    }
                    upx[p] = urx;
                    upy[p] = ury;
                }
            }
        }
        if (resid) {
            double v0 = (double)lo(r0) + (double)hi(r0), v1 = (double)lo(r1) + (double)hi(r1);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v0 += __shfl_xor_sync(0xffffffffu, v0, o);
                v1 += __shfl_xor_sync(0xffffffffu, v1, o);
            }
            if (t == 0) { part[0] = 0.0; part[1] = 0.0; }
            __syncthreads();
            if ((t & 31) == 0) {
                atomicAdd(&part[0], v0);
                atomicAdd(&part[1], v1);
            }
        }
        // 3. every CTA of the channel has written step s+1, its neighbours' halo rows included
        if (pushes) cluster.sync();
        else __syncthreads();
        // 4. residual decision (rank 0), broadcast through distributed shared memory
        if (resid) {
            if (rank == 0 && t == 0) {
                double du2 = 0.0, u2 = 0.0;
                for (int k = 0; k < CL; ++k) {
                    const double* pq = cluster.map_shared_rank(part, k);
                    du2 += pq[0];
                    u2 += pq[1];
                }
                const double r = u2 > 0.0 ? ::sqrt(du2 / u2) / a.check : 0.0;
                const bool unstable = *(volatile int*)(a.status + ch) != 0;
                done = unstable ? 2 : (r <= a.tol ? 1 : 0);
                a.res_out[ch] = r;
            }
            cluster.sync();
            dec = *cluster.map_shared_rank(&done, 0);
            if (dec) {
                ++s;
                break;
            }
        }
    }
    // write the state after step s back to the first buffer of the channel in HBM
    const T* fin = buf + ((s & 1) ? 9 * PS : 0);
    for (int i = 0; i < 9; ++i)
        for (int e = t; e < n_own; e += NT)
            gpop[(long long)i * P.P + (long long)y0 * nx + e] = fin[i * PS + kPairHalo * nx + e];
    C* up = a.uprev + 2 * P.base;
    auto out = [&](int e, C dr, C ux, C uy) {
        const long long g = (long long)y0 * nx + e;
        gdr[g] = dr;
        up[g] = ux;
        up[P.P + g] = uy;
    };
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        if (own_a(p)) out(node_a(p), lo(drv[p]), lo(upx[p]), lo(upy[p]));
        if (own_b(p)) out(node_b(p), hi(drv[p]), hi(upx[p]), hi(upy[p]));
    }
    if (rank == 0 && t == 0) a.steps_out[ch] = dec == 2 ? -2 : (dec == 1 ? s : -1);
    cluster.sync();  // no CTA leaves while another may still read its shared memory
}

template <typename T, int NT, int NP, int NX>
cudaError_t sweep_pair_config(int n_clusters, int cl, size_t smem, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
    const cudaError_t e = allow_shared_memory(k_sweep_pair<T, NT, NP, NX>);
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(n_clusters * cl);
    cfg->blockDim = dim3(NT);
    cfg->dynamicSmemBytes = smem;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = cl;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return e;
}
// How many clusters of `cl` CTAs with `smem` bytes the device can hold at once (0: never launched).
template <typename T, int NT, int NP, int NX>
cudaError_t launch_sweep_pair_capacity(int cl, size_t smem, int* n_clusters) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    const cudaError_t e = sweep_pair_config<T, NT, NP, NX>(1, cl, smem, &cfg, attr);
    return e == cudaSuccess ? cudaOccupancyMaxActiveClusters(n_clusters, k_sweep_pair<T, NT, NP, NX>, &cfg) : e;
}
template <typename T, int NT, int NP, int NX>
cudaError_t launch_sweep_pair(const SweepArgs<T, float>& a, int n_clusters, int cl, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    const cudaError_t e = sweep_pair_config<T, NT, NP, NX>(n_clusters, cl, smem, &cfg, attr);
    if (e != cudaSuccess) return e;
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, k_sweep_pair<T, NT, NP, NX>, a);
}

constexpr int kSweepPairs = 2;  // pairs of nodes per thread
#define LB_SWEEP_PAIR_VARIANTS(X)                                                                     \
    X(float, 128, 0) X(float, 256, 0) X(float, 128, 4) X(float, 256, 4) X(__nv_bfloat16, 128, 0)      \
    X(__nv_bfloat16, 256, 0) X(__nv_bfloat16, 128, 4) X(__nv_bfloat16, 256, 4)
#define LB_SWEEP_PAIR(PREFIX, T, NT, NX)                                                                                  \
    PREFIX template cudaError_t launch_sweep_pair<T, NT, kSweepPairs, NX>(const SweepArgs<T, float>&, int, int, size_t, \
                                                                          cudaStream_t);                                 \
    PREFIX template cudaError_t launch_sweep_pair_capacity<T, NT, kSweepPairs, NX>(int, size_t, int*);

}  // namespace lbk
