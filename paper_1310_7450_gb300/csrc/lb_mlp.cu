// lb_mlp.cu -- the learned warm start: a three-layer perceptron (n_in -> H -> H -> n_out, tanh on the
// hidden layers) trained and evaluated by this library's own kernels.  It maps channel parameters
// (width, body force, nlM parameters) to resampled steady profiles, which then initialise the
// lattice-Boltzmann run (lb_set_fields); the LB scheme stays the judge of the result.
//
// Numerics: the weights used by the forward and backward products are BF16 copies of FP32 master
// weights; every product accumulates in FP32; activations and gradients are FP32; Adam updates the
// FP32 masters and refreshes the BF16 copies.
//
// Layout: W1 [H][n_in], b1 [H], W2 [H][H], b2 [H], W3 [n_out][H], b3 [n_out], flattened in this
// order (lb_mlp_get_params / set_params / gradients use the same order).  Activations are row-major
// [batch][features].
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <new>
#include <vector>

#include "lbnlm.h"

namespace lbk {
void set_last_error(const char* msg);
}

namespace {

lb_status mfail(lb_status s, const char* what) {
    lbk::set_last_error(what);
    return s;
}
#define MLP_CK(call)                                                         \
    do {                                                                     \
        cudaError_t e_ = (call);                                             \
        if (e_ != cudaSuccess) {                                             \
            char m_[256];                                                    \
            std::snprintf(m_, sizeof m_, "%s: %s", #call, cudaGetErrorString(e_)); \
            return mfail(e_ == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA, m_); \
        }                                                                    \
    } while (0)

// ---- the products --------------------------------------------------------------------------------
// All of them are C[m][n] = sum_k A(m, k) B(k, n) in FP32, with what follows the product done where its
// sums are formed: the bias and tanh of a forward layer, the loss and its gradient behind the last one, the
// tanh' factor of a backward layer, Adam behind a weight gradient.
//
// A product is 17 to 50 million multiply-adds, 0.4 to 1.3 us of the part's FP32 rate: what bounds it is
// launching, reaching the operands in L2 and having enough CTAs, not arithmetic.  So a CTA takes a small tile
// (32 x 32, or 16 x 32 where that leaves fewer than one tile per SM), stages its operands over the whole depth at
// once, and splits the depth over groups of threads (8 or 16) that keep 4 x 4 sums per thread; the groups' sums are
// added in a fixed order in shared memory.  The launches of a step are five: the first layer (a few inputs)
// is evaluated where the second one stages its operand, and a weight gradient shares its launch with the
// input gradient of the layer below.  Each kernel is set up while the one before it drains (programmatic
// dependent launch) and stages what that one does not write; see Ready.
// 4 -> 256 -> 256 -> 768, us per training step / forward pass: batch 24 67.7 / 24.6 -> 25.2 / 9.8, 256 129.6 /
// 39.0 -> 43.5 / 20.6, 512 213 / 58 -> 68.7 / 26.2 (before: 16 x 16 tiles, 16-deep slabs, ten launches).
// 16 x 32 tiles at batch 256 take 48.7 / 21.5, 32 x 32 at 512 70.2 / 31.3 (the hidden layers' 128 tiles).
constexpr int kProdThreads = 512;
constexpr int kProdTn = 32;                          // tile width
constexpr int kFirstIn = 8;                          // inputs of a first layer evaluated inside the second
constexpr size_t kProdSmem = 200 * 1024;             // operand panels of one slab

enum Epilogue { EP_TANH, EP_LINEAR, EP_MSE, EP_DTANH, EP_GRAD };

// What a kernel may read before the grid before it in the stream has finished.  A kernel's blocks start when all
// blocks of that grid have passed their own wait, so the grids before that one have finished: the weights
// (written by the last launch of a step, or by the call before) are ready for every launch but the
// first, and an activation or gradient is when the grid that writes it lies two launches back.  Those grids have
// finished, so their results are in L2; that a kernel's L1 holds no older copy is promised only behind its own
// wait, so what is read ahead of it is loaded through L2 (ld.global.cg).
enum Ready { READY_NONE, READY_B, READY_ALL };  // READY_ALL: both operands; only the results wait

struct Adam {  // Adam (Kingma & Ba 2015) on the FP32 masters, then the BF16 working copy; p == nullptr: no update
    float *p, *m, *v;
    __nv_bfloat16* pb;
    float lr, b1, b2, eps, c1, c2;
};
// (pk, mk, vk: the element's parameter and moments, loaded ahead)
__device__ __forceinline__ void adam_update(const Adam& a, long long k, float gk, float pk, float mk, float vk) {
    mk = a.b1 * mk + (1.f - a.b1) * gk;
    vk = a.b2 * vk + (1.f - a.b2) * gk * gk;
    a.m[k] = mk;
    a.v[k] = vk;
    const float upd = a.lr * (mk / a.c1) / (sqrtf(vk / a.c2) + a.eps);
    pk = pk - upd;
    a.p[k] = pk;
    a.pb[k] = __float2bfloat16_rn(pk);
}

struct Product {
    const float* A;       // KMAJ: [m][k], else [k][m]
    const void* B;        // KMAJ: BF16 [n][k]; else BF16 or FP32 [k][n]
    float* C;             // [m][n] (EP_GRAD: null with Adam)
    int M, N, K;
    const float* bias;    // forward: [n]
    const float* aux;     // EP_DTANH: activations [m][n]; EP_MSE: targets [m][n]
    double* partial;      // EP_MSE: one sum of squares per tile
    float scale;          // EP_MSE: 1 / (number of outputs)
    float* bias_grad;     // EP_GRAD: row sums of A (null with Adam)
    Adam w, b;            // EP_GRAD: the weights' and the biases' update
    int tiles_n, tiles;
    int slab;             // depth staged at once
    // first layer evaluated in place of A (x != nullptr): A(m, k) = tanh(sum_i x[m][i] w1[k][i] + b1[k]),
    // also written to a1 by the first column of tiles
    const float* x;
    const __nv_bfloat16* w1;
    const float* b1;
    float* a1;
    int n_in;
};
// Wait for the grid before this one in the stream, and let the next one be set up.
__device__ __forceinline__ void grid_dependency() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// 16 bytes as FP32 values, and one value.  EARLY: of global memory ahead of the wait, through L2 (see Ready).
template <bool EARLY = false>
__device__ __forceinline__ void load16(const float* p, float (&v)[4]) {
    const float4 q = EARLY ? __ldcg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <bool EARLY = false>
__device__ __forceinline__ void load16(const __nv_bfloat16* p, float (&v)[8]) {
    const uint4* s = reinterpret_cast<const uint4*>(p);
    const uint4 q = EARLY ? __ldcg(s) : *s;  // (a BF16 value is the high half of its FP32 one)
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[2 * j] = __uint_as_float(w[j] << 16);
        v[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
}
template <bool EARLY>
__device__ __forceinline__ float load1(const float* p) { return EARLY ? __ldcg(p) : *p; }
template <bool EARLY>
__device__ __forceinline__ float load1(const __nv_bfloat16* p) {
    return __bfloat162float(EARLY ? __ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short*>(p))) : *p);
}

// Stage rows [r0, r0 + R) x depth [k0, k0 + kn) of an operand as dst[k][r] (row stride LD), zeros outside, in
// pieces of 16 bytes.  KMAJ: src[r][k] (depth contiguous): eight rows x four pieces per warp, which reads 64
// bytes of a row at a time and stores with few bank conflicts; else src[k][r].  U pieces per thread are on
// their way together.  (src is not __restrict__: read-only loads want data that no grid writes while this one
// exists, and the grid before it may still.)
template <bool EARLY, typename E, int R, int LD, bool KMAJ>
__device__ __forceinline__ void stage(float* dst, const E* src, int r0, int rows, int k0, int kn, int depth) {
    const int t = threadIdx.x;
    constexpr int V = 16 / (int)sizeof(E), U = sizeof(E) == 4 ? 6 : 4;
    const int kp = (kn + V - 1) / V;  // pieces along the depth
    const int pieces = KMAJ ? R * ((kp + 3) / 4 * 4) : kn * (R / V);
    const bool vec = (KMAJ ? depth : rows) % V == 0 && reinterpret_cast<uintptr_t>(src) % 16 == 0;
    for (int e0 = t; e0 < pieces; e0 += U * kProdThreads) {
        float v[U][V];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * kProdThreads;
#pragma unroll
            for (int j = 0; j < V; ++j) v[u][j] = 0.f;
            if (e >= pieces) continue;
            if constexpr (KMAJ) {
                const int r = (e & 7) + 8 * ((e >> 5) % (R / 8)), k = V * (((e >> 3) & 3) + 4 * ((e >> 5) / (R / 8)));
                if (k >= kn || r0 + r >= rows) continue;
                const E* p = src + (long long)(r0 + r) * depth + k0 + k;
                if (vec && k + V <= kn) load16<EARLY>(p, v[u]);
                else
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        if (k + j < kn) v[u][j] = load1<EARLY>(p + j);
            } else {
                const int r = V * (e % (R / V)), k = e / (R / V);
                const E* p = src + (long long)(k0 + k) * rows + r0 + r;
                if (vec && r0 + r + V <= rows) load16<EARLY>(p, v[u]);
                else
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        if (r0 + r + j < rows) v[u][j] = load1<EARLY>(p + j);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * kProdThreads;
            if (e >= pieces) continue;
            if constexpr (KMAJ) {
                const int r = (e & 7) + 8 * ((e >> 5) % (R / 8)), k = V * (((e >> 3) & 3) + 4 * ((e >> 5) / (R / 8)));
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (k + j < kn) dst[(k + j) * LD + r] = v[u][j];
            } else {
                const int r = V * (e % (R / V)), k = e / (R / V);
#pragma unroll
                for (int j = 0; j < V; j += 4)
                    *reinterpret_cast<float4*>(dst + k * LD + r + j) = make_float4(v[u][j], v[u][j + 1], v[u][j + 2], v[u][j + 3]);
            }
        }
    }
}

// One tile of a product.  TM: tile height; AK, BK: operand depth contiguous; E: type of B.
template <int TM, bool AK, bool BK, typename E, int EP, int READY, bool FIRST = false>
__device__ __forceinline__ void product_tile(const Product& q, int tile, float* smem) {
    constexpr int LA = TM + 4, LB = kProdTn + 4;
    constexpr int GT = (TM / 4) * (kProdTn / 4), G = kProdThreads / GT;  // threads per depth group, groups
    const int t = threadIdx.x, g = t / GT, l = t % GT;
    const int tn = 4 * (l % (kProdTn / 4)), tm = 4 * (l / (kProdTn / 4));
    const int m0 = (tile / q.tiles_n) * TM, n0 = (tile % q.tiles_n) * kProdTn;
    float* As = smem;
    float* Bs = smem + (size_t)q.slab * LA;
    const bool want_rows = EP == EP_GRAD && n0 == 0;  // (uniform) the row sums of A go with the first column of tiles
    float acc[4][4] = {}, rs[4] = {};
    // what the results need besides the sums: loaded ahead of the multiply-adds (pre[0]: bias, activation or
    // parameter; pre[1], pre[2]: target or Adam's moments)
    constexpr int OUT = TM * kProdTn / kProdThreads;
    float pre[OUT][3];
    for (int k0 = 0; k0 < q.K; k0 += q.slab) {
        const int kn = min(q.slab, q.K - k0);
        if (k0) __syncthreads();
        if (READY == READY_NONE && k0 == 0) grid_dependency();
        stage<READY != READY_NONE, E, kProdTn, LB, BK>(Bs, static_cast<const E*>(q.B), n0, q.N, k0, kn, q.K);
        if (READY == READY_B && k0 == 0) grid_dependency();
        if constexpr (FIRST) {  // (one slab: k0 = 0, kn = K)
            // the first layer's weights as FP32 rows of kFirstIn, zero-padded; a thread keeps one row of x
            float* ws = smem + (size_t)q.slab * (LA + LB);
            for (int e = t; e < kn * kFirstIn; e += kProdThreads) {
                const int i = e % kFirstIn, k = e / kFirstIn;
                ws[e] = i < q.n_in ? __bfloat162float(q.w1[(long long)k * q.n_in + i]) : 0.f;
            }
            float* b1 = ws + kn * kFirstIn;
            for (int k = t; k < kn; k += kProdThreads) b1[k] = q.b1[k];
            const int r = t % TM;
            float x[kFirstIn];
#pragma unroll
            for (int i = 0; i < kFirstIn; ++i)
                x[i] = i < q.n_in && m0 + r < q.M ? q.x[(long long)(m0 + r) * q.n_in + i] : 0.f;
            __syncthreads();
#pragma unroll 2
            for (int k = t / TM; k < kn; k += kProdThreads / TM) {
                float w0[4], w1[4], v = 0.f;
                load16(ws + k * kFirstIn, w0);
                load16(ws + k * kFirstIn + 4, w1);
#pragma unroll
                for (int i = 0; i < 4; ++i) v = fmaf(x[i], w0[i], v);
#pragma unroll
                for (int i = 0; i < 4; ++i) v = fmaf(x[4 + i], w1[i], v);
                As[k * LA + r] = m0 + r < q.M ? tanhf(v + b1[k]) : 0.f;
            }
            if (n0 == 0) {
                __syncthreads();
                for (int e = t; e < TM * kn; e += kProdThreads)
                    if (m0 + e / kn < q.M) q.a1[(long long)(m0 + e / kn) * kn + e % kn] = As[(e % kn) * LA + e / kn];
            }
        } else {
            stage<READY == READY_ALL, float, TM, LA, AK>(As, q.A, m0, q.M, k0, kn, q.K);
        }
        if (k0 == 0)
#pragma unroll
            for (int u = 0; u < OUT; ++u) {
                const int e = t + u * kProdThreads, m = m0 + e / kProdTn, n = n0 + e % kProdTn;
                pre[u][0] = pre[u][1] = pre[u][2] = 0.f;
                if (m >= q.M || n >= q.N) continue;
                const long long o = (long long)m * q.N + n;
                if constexpr (EP == EP_TANH || EP == EP_LINEAR || EP == EP_MSE) pre[u][0] = q.bias[n];
                if constexpr (EP == EP_MSE) pre[u][1] = q.aux[o];
                if constexpr (EP == EP_DTANH) pre[u][0] = q.aux[o];
                if constexpr (EP == EP_GRAD)
                    if (q.w.p) { pre[u][0] = __ldcg(q.w.p + o); pre[u][1] = __ldcg(q.w.m + o); pre[u][2] = __ldcg(q.w.v + o); }
            }
        __syncthreads();
        const int per = (kn + G - 1) / G, ka = g * per, kb = min(kn, ka + per);
#pragma unroll 8
        for (int k = ka; k < kb; ++k) {
            float a[4], b[4];
            load16(As + k * LA + tm, a);
            load16(Bs + k * LB + tn, b);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            if (want_rows)
#pragma unroll
                for (int i = 0; i < 4; ++i) rs[i] += a[i];
        }
    }
    // the groups' sums, added in the groups' order
    __syncthreads();
    float* red = smem;                       // [G][TM][kProdTn]
    float* rred = smem + G * TM * kProdTn;   // [G][TM]
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(red + (g * TM + tm + i) * kProdTn + tn) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (want_rows && tn == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) rred[g * TM + tm + i] = rs[i];
    __syncthreads();
    if (READY == READY_ALL) grid_dependency();
    double sq = 0.0;
#pragma unroll
    for (int u = 0; u < OUT; ++u) {
        const int e = t + u * kProdThreads, m = m0 + e / kProdTn, n = n0 + e % kProdTn;
        if (m >= q.M || n >= q.N) continue;
        float v = red[e];
#pragma unroll
        for (int k = 1; k < G; ++k) v += red[k * TM * kProdTn + e];
        const long long o = (long long)m * q.N + n;
        if constexpr (EP == EP_TANH) q.C[o] = tanhf(v + pre[u][0]);
        if constexpr (EP == EP_LINEAR) q.C[o] = v + pre[u][0];
        if constexpr (EP == EP_MSE) {  // loss = mean (y - t)^2, C = 2 (y - t) / n
            const float d = v + pre[u][0] - pre[u][1];
            q.C[o] = 2.f * d * q.scale;
            sq += (double)d * d;
        }
        if constexpr (EP == EP_DTANH) q.C[o] = v * (1.f - pre[u][0] * pre[u][0]);
        if constexpr (EP == EP_GRAD) {
            if (q.w.p) adam_update(q.w, o, v, pre[u][0], pre[u][1], pre[u][2]);
            else q.C[o] = v;
        }
    }
    if (want_rows && t < TM && m0 + t < q.M) {
        float v = rred[t];
        for (int k = 1; k < G; ++k) v += rred[k * TM + t];
        if (q.b.p) adam_update(q.b, m0 + t, v, q.b.p[m0 + t], q.b.m[m0 + t], q.b.v[m0 + t]);
        else q.bias_grad[m0 + t] = v;
    }
    if constexpr (EP == EP_MSE) {
        __syncthreads();
        double* dred = reinterpret_cast<double*>(smem);
        dred[t] = sq;   // (two FP64 additions per SM and clock: one warp adds, not sixteen)
        __syncthreads();
        if (t < 32) {
            for (int k = t + 32; k < kProdThreads; k += 32) sq += dred[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (t == 0) q.partial[tile] = sq;
        }
    }
}

// (two CTAs per SM, 64 registers, where the compiler would take 72: a step at batch 2048 241 -> 224 us, at 256 46.8 ->
// 43.7; it does not change the other layers')
template <int TM, int EP, int READY, bool FIRST>
__global__ void __launch_bounds__(kProdThreads, EP == EP_MSE || FIRST ? 2 : 0) k_forward(const Product q) {
    extern __shared__ __align__(16) float prod_smem[];
    product_tile<TM, true, true, __nv_bfloat16, EP, READY, FIRST>(q, blockIdx.x, prod_smem);
}
// input gradient of one layer (x) and weight gradient of the layer above (w, whose operands are older)
template <int TX, int TW>
__global__ void __launch_bounds__(kProdThreads) k_backward(const Product x, const Product w) {
    extern __shared__ __align__(16) float prod_smem[];
    if ((int)blockIdx.x < x.tiles) product_tile<TX, true, false, __nv_bfloat16, EP_DTANH, READY_B>(x, blockIdx.x, prod_smem);
    else product_tile<TW, false, false, float, EP_GRAD, READY_ALL>(w, blockIdx.x - x.tiles, prod_smem);
}
// the weight gradients of the lower two layers (b: the first layer's, of the gradient just formed)
template <int TA, int TB>
__global__ void __launch_bounds__(kProdThreads) k_weights(const Product a, const Product b) {
    extern __shared__ __align__(16) float prod_smem[];
    if ((int)blockIdx.x < b.tiles) product_tile<TB, false, false, float, EP_GRAD, READY_NONE>(b, blockIdx.x, prod_smem);
    else product_tile<TA, false, false, float, EP_GRAD, READY_ALL>(a, blockIdx.x - b.tiles, prod_smem);
}

// Tile height and tiles of a product; returns its shared memory.
int tile_height(int M, int N) {
    const int n = (N + kProdTn - 1) / kProdTn;
    return (long long)((M + 31) / 32) * n >= 152 ? 32 : 16;
}
size_t plan(Product& q, int tm) {
    q.tiles_n = (q.N + kProdTn - 1) / kProdTn;
    q.tiles = (q.M + tm - 1) / tm * q.tiles_n;
    const int row = (tm + 4 + kProdTn + 4) * (int)sizeof(float);
    q.slab = std::min(q.K, (int)(kProdSmem / row) / 8 * 8);
    const int G = kProdThreads / ((tm / 4) * (kProdTn / 4));
    return std::max((size_t)q.slab * row, (size_t)G * tm * (kProdTn + 1) * sizeof(float));
}
// Once per handle, on its device: every product kernel may take its shared memory.
cudaError_t allow_shared_memory() {
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto k) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProdSmem);
    };
    allow(k_forward<16, EP_TANH, READY_NONE, true>);
    allow(k_forward<32, EP_TANH, READY_NONE, true>);
    allow(k_forward<16, EP_TANH, READY_NONE, false>);
    allow(k_forward<32, EP_TANH, READY_NONE, false>);
    allow(k_forward<16, EP_TANH, READY_B, false>);
    allow(k_forward<32, EP_TANH, READY_B, false>);
    allow(k_forward<16, EP_LINEAR, READY_B, false>);
    allow(k_forward<32, EP_LINEAR, READY_B, false>);
    allow(k_forward<16, EP_MSE, READY_B, false>);
    allow(k_forward<32, EP_MSE, READY_B, false>);
    allow(k_backward<16, 32>);
    allow(k_weights<16, 16>);
    return e;
}
template <typename K, typename... Args>
cudaError_t launch(K k, int grid, size_t smem, cudaStream_t s, const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kProdThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

__global__ void k_to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ pb, long long n) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        pb[k] = __float2bfloat16_rn(p[k]);
}

// Deterministic initialisation (uniform in +-1/sqrt(fan_in), SplitMix64 bits), biases zero.
__global__ void k_init_params(float* __restrict__ p, long long off, long long n, int fan_in, unsigned long long seed) {
    const float a = rsqrtf((float)fan_in);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        unsigned long long z = seed + (unsigned long long)(off + k + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const float u = (float)((double)(z >> 11) * 0x1p-53) * 2.f - 1.f;
        p[off + k] = a * u;
    }
}

int nblocks(long long n) {
    long long b = (n + 255) / 256;
    return (int)(b < 1 ? 1 : (b > 2048 ? 2048 : b));
}

}  // namespace

struct lb_mlp {
    int n_in = 0, H = 0, n_out = 0, max_batch = 0;
    int dev = 0;  // device that was current at creation
    cudaStream_t stream = nullptr;
    long long n_par = 0, o_w1 = 0, o_b1 = 0, o_w2 = 0, o_b2 = 0, o_w3 = 0, o_b3 = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // masters, gradients, Adam moments
    __nv_bfloat16* pb = nullptr;                                    // BF16 working weights
    float *a1 = nullptr, *a2 = nullptr, *y = nullptr;              // activations [max_batch][..]
    float *d1 = nullptr, *d2 = nullptr, *dy = nullptr;             // their gradients
    double* partial = nullptr;                                      // loss partial sums, one per tile
    long long t = 0;                                                // Adam step
};

namespace {

void mlp_free(lb_mlp* m) {
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    for (void* q : {(void*)m->p, (void*)m->g, (void*)m->m, (void*)m->v, (void*)m->pb, (void*)m->a1, (void*)m->a2,
                    (void*)m->y, (void*)m->d1, (void*)m->d2, (void*)m->dy, (void*)m->partial})
        if (q) cudaFree(q);
    delete m;
}

template <int EP, int READY, bool FIRST = false>
cudaError_t run_forward(lb_mlp* m, Product q) {
    const int tm = tile_height(q.M, q.N);
    const size_t smem = plan(q, tm) + (FIRST ? sizeof(float) * (kFirstIn + 1) * q.K : 0);
    return tm == 32 ? launch(k_forward<32, EP, READY, FIRST>, q.tiles, smem, m->stream, q)
                    : launch(k_forward<16, EP, READY, FIRST>, q.tiles, smem, m->stream, q);
}

Product forward_product(lb_mlp* m, const float* in, long long o_w, long long o_b, float* out, int B, int I, int O) {
    Product q{};
    q.A = in;
    q.B = m->pb + o_w;
    q.C = out;
    q.M = B;
    q.N = O;
    q.K = I;
    q.bias = m->p + o_b;
    return q;
}

// The two hidden layers: in one launch when the first has few inputs (every tile of the second evaluates its
// rows of the first again) and the second's depth fits one slab.
lb_status forward_hidden(lb_mlp* m, const float* x, int B) {
    Product q = forward_product(m, m->a1, m->o_w2, m->o_b2, m->a2, B, m->H, m->H);
    if (m->n_in <= kFirstIn && plan(q, 32) + sizeof(float) * (kFirstIn + 1) * m->H <= kProdSmem && q.slab == m->H) {
        q.x = x;
        q.w1 = m->pb + m->o_w1;
        q.b1 = m->p + m->o_b1;
        q.a1 = m->a1;
        q.n_in = m->n_in;
        MLP_CK((run_forward<EP_TANH, READY_NONE, true>(m, q)));
    } else {
        MLP_CK((run_forward<EP_TANH, READY_NONE>(m, forward_product(m, x, m->o_w1, m->o_b1, m->a1, B, m->n_in, m->H))));
        MLP_CK((run_forward<EP_TANH, READY_B>(m, q)));
    }
    return LB_OK;
}

lb_status forward(lb_mlp* m, const float* x, int B, float* y) {
    lb_status st = forward_hidden(m, x, B);
    if (st != LB_OK) return st;
    MLP_CK((run_forward<EP_LINEAR, READY_B>(m, forward_product(m, m->a2, m->o_w3, m->o_b3, y, B, m->H, m->n_out))));
    return LB_OK;
}

// dX[b][i] = sum_o dY[b][o] W[o][i] times tanh' of the input's activations
Product input_gradient(lb_mlp* m, const float* dy, long long o_w, const float* act, float* dx, int B, int I, int O) {
    Product q{};
    q.A = dy;
    q.B = m->pb + o_w;
    q.C = dx;
    q.M = B;
    q.N = I;
    q.K = O;
    q.aux = act;
    return q;
}
// dW[o][i] = sum_b dY[b][o] X[b][i] and db[o] = sum_b dY[b][o]: into m->g, or Adam's update of the layer
Product weight_gradient(lb_mlp* m, const float* dy, const float* x, long long o_w, long long o_b, int B, int I, int O,
                        const Adam* adam) {
    Product q{};
    q.A = dy;
    q.B = x;
    q.M = O;
    q.N = I;
    q.K = B;
    if (adam) {
        auto at = [&](long long o) {
            Adam a = *adam;
            a.p = m->p + o;
            a.m = m->m + o;
            a.v = m->v + o;
            a.pb = m->pb + o;
            return a;
        };
        q.w = at(o_w);
        q.b = at(o_b);
    } else {
        q.C = m->g + o_w;
        q.bias_grad = m->g + o_b;
    }
    return q;
}

// Forward, loss and the full gradient: into m->g, or (adam) straight into the update of the parameters.  A layer's
// weights change in a launch after the one whose input gradient reads them.  The loss (host) if
// requested.
lb_status backward(lb_mlp* m, const float* x, const float* target, int B, double* loss, const Adam* adam) {
    lb_status st = forward_hidden(m, x, B);
    if (st != LB_OK) return st;
    const long long n = (long long)B * m->n_out;
    Product y = forward_product(m, m->a2, m->o_w3, m->o_b3, m->dy, B, m->H, m->n_out);
    y.aux = target;
    y.partial = m->partial;
    y.scale = 1.f / (float)n;
    const int ty = tile_height(y.M, y.N);
    plan(y, ty);
    MLP_CK((run_forward<EP_MSE, READY_B>(m, y)));
    Product none{};
    Product x3 = input_gradient(m, m->dy, m->o_w3, m->a2, m->d2, B, m->H, m->n_out);
    Product x2 = input_gradient(m, m->d2, m->o_w2, m->a1, m->d1, B, m->H, m->H);
    Product w3 = weight_gradient(m, m->dy, m->a2, m->o_w3, m->o_b3, B, m->H, m->n_out, adam);
    Product w2 = weight_gradient(m, m->d2, m->a1, m->o_w2, m->o_b2, B, m->H, m->H, adam);
    Product w1 = weight_gradient(m, m->d1, x, m->o_w1, m->o_b1, B, m->n_in, m->H, adam);
    size_t smem = plan(x3, 16);
    MLP_CK(launch(k_backward<16, 32>, x3.tiles, smem, m->stream, x3, none));
    smem = std::max(plan(x2, 16), plan(w3, 32));
    MLP_CK(launch(k_backward<16, 32>, x2.tiles + w3.tiles, smem, m->stream, x2, w3));
    smem = std::max(plan(w2, 16), plan(w1, 16));
    MLP_CK(launch(k_weights<16, 16>, w2.tiles + w1.tiles, smem, m->stream, w2, w1));
    if (loss) {
        std::vector<double> part(y.tiles);
        MLP_CK(cudaMemcpyAsync(part.data(), m->partial, sizeof(double) * y.tiles, cudaMemcpyDeviceToHost, m->stream));
        MLP_CK(cudaStreamSynchronize(m->stream));
        double s = 0.0;
        for (double q : part) s += q;
        *loss = s / (double)n;
    }
    return LB_OK;
}

}  // namespace

extern "C" {

lb_status lb_mlp_create(int n_in, int width, int n_out, int max_batch, uint64_t seed, void* cuda_stream, lb_mlp** out) {
    if (!out) return mfail(LB_EINVAL, "lb_mlp_create: out is null");
    *out = nullptr;
    if (n_in < 1 || width < 1 || n_out < 1 || max_batch < 1) return mfail(LB_EINVAL, "lb_mlp_create: sizes must be >= 1");
    lb_mlp* m = new (std::nothrow) lb_mlp();
    if (!m) return mfail(LB_ENOMEM, "lb_mlp_create: host allocation");
    m->n_in = n_in; m->H = width; m->n_out = n_out; m->max_batch = max_batch;
    m->stream = (cudaStream_t)cuda_stream;
    cudaGetDevice(&m->dev);
    m->o_w1 = 0; m->o_b1 = m->o_w1 + (long long)width * n_in;
    m->o_w2 = m->o_b1 + width; m->o_b2 = m->o_w2 + (long long)width * width;
    m->o_w3 = m->o_b2 + width; m->o_b3 = m->o_w3 + (long long)n_out * width;
    m->n_par = m->o_b3 + n_out;
    const long long P = m->n_par, B = max_batch;
    cudaError_t e = cudaSuccess;
    auto al = [&](void** q, size_t bytes) { if (e == cudaSuccess) e = cudaMalloc(q, bytes); };
    al((void**)&m->p, P * 4); al((void**)&m->g, P * 4); al((void**)&m->m, P * 4); al((void**)&m->v, P * 4);
    al((void**)&m->pb, P * 2);
    al((void**)&m->a1, B * width * 4); al((void**)&m->a2, B * width * 4); al((void**)&m->y, B * n_out * 4);
    al((void**)&m->d1, B * width * 4); al((void**)&m->d2, B * width * 4); al((void**)&m->dy, B * n_out * 4);
    al((void**)&m->partial, (size_t)((B + 15) / 16) * ((n_out + kProdTn - 1) / kProdTn) * sizeof(double));
    if (e != cudaSuccess) { mlp_free(m); return mfail(LB_ENOMEM, "lb_mlp_create: cudaMalloc"); }
    if (allow_shared_memory() != cudaSuccess) { mlp_free(m); return mfail(LB_ECUDA, "lb_mlp_create: kernel attributes"); }
    e = cudaMemsetAsync(m->p, 0, P * 4, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, P * 4, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, P * 4, m->stream);
    if (e != cudaSuccess) { mlp_free(m); return mfail(LB_ECUDA, "lb_mlp_create: memset"); }
    k_init_params<<<nblocks(m->o_b1), 256, 0, m->stream>>>(m->p, m->o_w1, m->o_b1 - m->o_w1, n_in, seed);
    k_init_params<<<nblocks(m->o_b2 - m->o_w2), 256, 0, m->stream>>>(m->p, m->o_w2, m->o_b2 - m->o_w2, width, seed ^ 0x5bd1e995ull);
    k_init_params<<<nblocks(m->o_b3 - m->o_w3), 256, 0, m->stream>>>(m->p, m->o_w3, m->o_b3 - m->o_w3, width, seed ^ 0x27d4eb2full);
    k_to_bf16<<<nblocks(P), 256, 0, m->stream>>>(m->p, m->pb, P);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) { mlp_free(m); return mfail(LB_ECUDA, "lb_mlp_create: init kernels"); }
    *out = m;
    return LB_OK;
}

void lb_mlp_destroy(lb_mlp* m) { mlp_free(m); }

long long lb_mlp_num_params(const lb_mlp* m) { return m ? m->n_par : 0; }

lb_status lb_mlp_forward(lb_mlp* m, const float* x, int batch, float* y) {
    if (!m || !x || !y || batch < 1 || batch > m->max_batch) return mfail(LB_EINVAL, "lb_mlp_forward: bad argument");
    // this device's memory is written by the last layer itself; anything else (another device's memory, an address
    // that is no multiple of 4) gets a copy
    cudaPointerAttributes at{};
    const bool direct = (uintptr_t)y % sizeof(float) == 0 && cudaPointerGetAttributes(&at, y) == cudaSuccess &&
                        ((at.type == cudaMemoryTypeDevice && at.device == m->dev) || at.type == cudaMemoryTypeManaged);
    (void)cudaGetLastError();
    lb_status st = forward(m, x, batch, direct ? y : m->y);
    if (st != LB_OK || direct) return st;
    MLP_CK(cudaMemcpyAsync(y, m->y, sizeof(float) * batch * m->n_out, cudaMemcpyDeviceToDevice, m->stream));
    return LB_OK;
}

lb_status lb_mlp_gradients(lb_mlp* m, const float* x, const float* target, int batch, float* grads, double* loss) {
    if (!m || !x || !target || batch < 1 || batch > m->max_batch) return mfail(LB_EINVAL, "lb_mlp_gradients: bad argument");
    lb_status st = backward(m, x, target, batch, loss, nullptr);
    if (st != LB_OK) return st;
    if (grads) MLP_CK(cudaMemcpyAsync(grads, m->g, sizeof(float) * m->n_par, cudaMemcpyDeviceToDevice, m->stream));
    return LB_OK;
}

lb_status lb_mlp_train_step(lb_mlp* m, const float* x, const float* target, int batch, float lr, double* loss) {
    if (!m || !x || !target || batch < 1 || batch > m->max_batch || !(lr > 0.f))
        return mfail(LB_EINVAL, "lb_mlp_train_step: bad argument");
    Adam adam{};
    const float t = (float)(m->t + 1);
    adam.lr = lr;
    adam.b1 = 0.9f;
    adam.b2 = 0.999f;
    adam.eps = 1e-8f;
    adam.c1 = 1.f - powf(adam.b1, t);
    adam.c2 = 1.f - powf(adam.b2, t);
    lb_status st = backward(m, x, target, batch, loss, &adam);
    if (st == LB_OK) m->t += 1;
    return st;
}

lb_status lb_mlp_get_params(lb_mlp* m, float* host) {
    if (!m || !host) return mfail(LB_EINVAL, "lb_mlp_get_params: null argument");
    MLP_CK(cudaMemcpyAsync(host, m->p, sizeof(float) * m->n_par, cudaMemcpyDeviceToHost, m->stream));
    MLP_CK(cudaStreamSynchronize(m->stream));
    return LB_OK;
}

lb_status lb_mlp_set_params(lb_mlp* m, const float* host) {
    if (!m || !host) return mfail(LB_EINVAL, "lb_mlp_set_params: null argument");
    MLP_CK(cudaMemcpyAsync(m->p, host, sizeof(float) * m->n_par, cudaMemcpyHostToDevice, m->stream));
    k_to_bf16<<<nblocks(m->n_par), 256, 0, m->stream>>>(m->p, m->pb, m->n_par);
    MLP_CK(cudaGetLastError());
    MLP_CK(cudaStreamSynchronize(m->stream));
    return LB_OK;
}

}  // extern "C"
