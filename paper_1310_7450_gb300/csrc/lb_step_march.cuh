// lb_step_march.cuh -- the fused lattice-Boltzmann step for wide channels: a TMA-fed row march.
//
// A CTA owns a strip of CW columns (x0 .. x0+CW-1), two adjacent columns per thread, and marches
// through rows y0..y1-1 of one channel.  The post-collision populations of the previous step stream into a
// ring of K shared-memory slots, one source row per slot: a single 3-D tensor-memory-access copy
// brings the 9 direction planes of that row, columns x0-HP .. x0+CW+HP-1 (HP = 16 bytes of halo on each
// side, so every copy starts on a 16-byte boundary).  The copies run K-2 rows ahead of the arithmetic
// and complete on one mbarrier per slot.
//
// Per row y (one __syncthreads per row):
//   1. moments (Eq. rhoj) of row y+1 for the own columns and the two halo columns x0-1, x0+CW,
//      pulled from slots y, y+1, y+2 (Eq. lbupdate, pull form; bounce-back at the walls,
//      Sec. II B); the own populations and gradient velocities j/R0 stay in registers, and what the
//      neighbouring threads need of the velocities goes through shuffles or shared memory;
//   2. barrier; one thread (the last lane) refills the slot of row y with row y+K;
//   3. collision of row y: kappa by three-point differences (along y from the thread's own
//      registers), the nlM stress, Sigma^nN, delta rho, n^eq, F_i
//      (Eq. bodyforce), BGK; coalesced stores (8-byte FP32 pairs, 4-byte BF16 pairs).
// The two columns of a thread go through the arithmetic together as packed FP32 (lb_pair.cuh).
// The periodic wrap of x is patched into the halo columns of the first and last strip with
// plain loads.  Every mbarrier wait is bounded (MarchCtl::max_wait_ns, 2 s by default): on timeout
// the CTA records LB_ETIMEOUT in the status word, drains its own copies (also bounded) and returns.
#pragma once

#include <cuda.h>

#include "lb_march_plan.h"
#include "lb_pair.cuh"

namespace lbk {

enum : int { kFull = 0, kPart = 1, kOdd = 2 };  // strips of a channel, see k_step_march

struct MarchCtl {
    const MarchItem* items;
    int n_items;
    int* timeout_flag;  // the channel status word: bit 2 is set when a bounded wait gave up
    long long plane;    // plane stride of the channel's fields (elements)
    long long base;     // plane offset of the channel (its planes start at k * base)
    unsigned long long max_wait_ns;  // limit of every mbarrier wait (0: one non-blocking probe)
    // the last CTA to finish (done_count counts them; zero between launches) stores the channel's
    // status word into status_host (mapped pinned host memory: the host polls it without a copy
    // in the stream) and, on monitor steps (mon set), reduces the item partials into mon[0..3]
    unsigned* done_count = nullptr;
    int* status_host = nullptr;
    double* mon = nullptr;
    long long state_index = 0;
    int with_residual = 0;
    bool dependent = false;  // host: programmatic dependent launch
};

// A CTA whose wait gave up waits this long for its own copies in flight before it returns.  A
// bulk copy that has not landed after a second means the memory system has failed; the CTA
// leaves then rather than spin without end.
constexpr unsigned long long kMarchDrainNs = 1000000000ull;

// ---- PTX helpers (mbarrier, TMA) ----------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for the phase with the given parity: mbarrier.try_wait suspends the thread until
// the phase completes or a hardware time limit passes; the loop gives up after max_ns of wall
// time (returns false then).  max_ns = 0: a single non-blocking probe (mbarrier.test_wait).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t max_ns) {
    const uint32_t a = smem_u32(bar);
    if (max_ns == 0) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        return done != 0;
    }
    uint64_t t0 = 0;
    for (uint32_t k = 0;; ++k) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if (k == 0) t0 = global_ns();
        else if (global_ns() - t0 > max_ns) return false;
    }
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}
// Bulk prefetch of bytes (a multiple of 16, 16-byte aligned) from global memory into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

template <typename T>
struct MarchGeom {
    static constexpr int HP = 16 / (int)sizeof(T);  // halo columns per side (16 bytes)
};

// Elements of a slot row: the strip and its halo; ODD: and up to HP - 1 elements before them, since a copy starts
// on a 16-byte boundary and the rows of a channel whose width is no multiple of 16 bytes do not.
template <typename T>
__host__ __device__ constexpr int march_slot_width(int W, bool odd) { return W + (odd ? 3 : 2) * MarchGeom<T>::HP; }

// Shared-memory footprint of the march kernel (bytes).
template <typename T, typename C, int W, int K, bool ODD>
constexpr size_t march_smem_bytes() {
    constexpr size_t slot = ((size_t)9 * march_slot_width<T>(W, ODD) * sizeof(T) + 8 + 127) / 128 * 128;
    return K * slot + (std::is_same<T, float>::value ? (size_t)W * 2 * sizeof(C) + 4 * 4 * 2 * sizeof(C)
                                                     : (size_t)4 * (W + 4) * 2 * sizeof(C));
}

// Rows of a field of the arithmetic type: the thread's two adjacent columns as one 8-byte access.
__device__ __forceinline__ P2 load_pair(const float* p) {
    P2 r;
    r.v = *reinterpret_cast<const unsigned long long*>(p);
    return r;
}
__device__ __forceinline__ void store_pair(float* p, P2 v) { *reinterpret_cast<unsigned long long*>(p) = v.v; }
// Populations in the storage type: FP32 as above; BF16 rounded to nearest, one 4-byte store.
__device__ __forceinline__ void store_pop_pair(float* p, P2 v) { store_pair(p, v); }
__device__ __forceinline__ void store_pop_pair(__nv_bfloat16* p, P2 v) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(lo(v), hi(v));
}
// Two neighbouring populations of a slot row, as FP32: at an even column one access, at an odd one two.
__device__ __forceinline__ P2 slot_pair(const float* p) { return load_pair(p); }
__device__ __forceinline__ P2 slot_pair(const __nv_bfloat16* p) {
    const uint32_t w = *reinterpret_cast<const uint32_t*>(p);  // (a BF16 value is the high half of its FP32 one)
    return p2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
template <typename T>
__device__ __forceinline__ P2 slot_pair_odd(const T* p) {
    return p2((float)Store<T>::cvt(p[0]), (float)Store<T>::cvt(p[1]));
}

// BND = 1: channel ends joined by the generalized periodic boundaries of Sec. II B, and a moving
// Couette wall on the last row (Sec. IV C) if the channel has one; BND = 2: the moving wall only;
// both applied where the populations are pulled (the same rules as the tile kernel's pull9).
// BND = 0: periodic x and bounce-back walls only.
// SCHEME 1: the generalized-Newtonian comparison scheme of Sec. II C (periodic x, bounce-back
// walls, stress mode A), the node's own relaxation rate as in the tile kernel's scheme-1 variant.
// SCHEME 3: the relaxation-time extensions (periodic x, bounce-back walls, either stress mode): the
// node's FP64 fluidity is loaded one row ahead of its use and stored with the step, as in the tile
// kernel's scheme-3 variant.
// STRIP: kFull, the width is a multiple of CW; kPart, strips of another width, rows a multiple of 16 bytes; kOdd,
// rows of any length.  kOdd's copies come from a map of the planes as one long row each, start on the
// 16-byte boundary before the strip, and the pulls add the remainder of each row; its global loads and
// stores go column by column.  (Variants of their own: the masks of a partial strip cost whole strips 13 % in
// FP32 and 22 % in BF16.)
// FIELDS: the fields of the stored state (F_FIELDS) instead of a step: everything up to the stress, then
// u, sigma and rho in node order.
template <typename T, typename C, int SMODE, int CW, int K, int BND = 0, int SCHEME = 0, bool FIELDS = false, int STRIP = 0>
__global__ void __launch_bounds__(CW / 2, 6) k_step_march(const __grid_constant__ CUtensorMap tmap,
                                                                                  const StepArgs<T, C> a,
                                                                                  const MarchCtl ctl) {
    static_assert(std::is_same<C, float>::value, "the pair arithmetic is FP32");
    constexpr int NT = CW / 2;                                       // threads per CTA
    constexpr bool ODD = STRIP == kOdd;
    constexpr int HP = MarchGeom<T>::HP;
    constexpr int SW = march_slot_width<T>(CW, ODD);                 // slot row width (elements)
    constexpr uint32_t TX = 9u * SW * sizeof(T);                     // bytes per copy
    constexpr uint32_t SLOT = (TX + 8 + 127) / 128 * 128;            // a slot: the copy, then its mbarrier
    // measured choices, see the note above the launchers
    constexpr bool F32 = std::is_same<T, float>::value;
    constexpr bool HALO2 = BND != 1 || !F32;    // both halo columns of two rows in one pass
    constexpr bool UNROLL2 = BND != 1 || !F32;  // the row loop written out for two rows
    constexpr bool SHUFFLE = F32;      // neighbouring columns' velocities by warp shuffles, or a ring of rows
    constexpr bool OFF32 = F32;
    constexpr int UW = CW + 4;         // ring row: columns x0-2 .. x0+CW+1
    static_assert(NT == 64, "two warps: the border velocities, the edge patchers, the issuing thread");

    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* slots = smem;                                      // K slots
    // own velocities of the row two rows from a wall (the one-sided difference of the wall row), and
    // per row (ring of 4) the velocities that cross a warp's border: x0-1, the border columns, x0+CW
    // (SHUFFLE), or a ring of 4 rows of velocity pairs, two columns of one thread on a 16-byte boundary
    C* uwall = reinterpret_cast<C*>(slots + K * SLOT);                // SHUFFLE: [CW][2]
    float2* edge = reinterpret_cast<float2*>(uwall + 2 * CW);         // SHUFFLE: [4][4]
    auto ring = [&](int r, int col) -> C* { return uwall + 2 * ((r & 3) * UW + col + 2); };

    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;

    __shared__ int s_bad;  // set by any thread whose bounded wait gave up; read after a barrier
    __shared__ C s_delta[2];  // BND == 1 with GPBC: rho_out - mean(x = 0), rho_in - mean(x = nx-1)
    // BND == 1 with GPBC: the bracket of the end-crossing rebuild (gpbc_shift_core) of every
    // population that leaves a boundary column across the end, per source row (ring of 8 rows),
    // boundary column c (0: x = 0, directions 3, 6, 7; 1: x = nx-1, directions 1, 5, 8) and
    // direction; six lanes of an edge strip fill one row, the pulls read it
    __shared__ C s_shift[BND == 1 ? 8 : 1][2][3];
    constexpr int TI = NT - 1;  // the thread that issues the copies (last lane; warp 0 computes
                                // the halo columns)
    constexpr int TP = NT - 2;  // the thread that issues the L2 prefetches of residual steps
    auto bar_at = [&](uint32_t off) -> uint64_t* { return reinterpret_cast<uint64_t*>(slots + off + TX); };
    if (t == 0) {
        s_bad = 0;
        prefetch_tmap(&tmap);
        for (int k = 0; k < K; ++k) mbar_init(bar_at(k * SLOT), 1);
        fence_barrier_init();
    }
    grid_dependency();
    const ChanParams<C> P = a.chan[0];
    const int nx = a.nx, ny = P.ny;
    const bool halted = a.status[0] != 0;  // an unstable or timed-out channel takes no more steps
    if (BND == 1 && t == 0 && a.gcol != nullptr) {
        const C* means = a.gcol + 6LL * a.gny;  // [channel][column] means of rho - 1
        s_delta[0] = P.rho_out - means[0];
        s_delta[1] = P.rho_in - means[1];
    }
    __syncthreads();

    const PairConst q = pair_const(P);
    bool vbad = false;  // some node of this CTA failed the velocity guard (reported when the CTA ends)
    uint32_t nload = 0;  // CTA-uniform count of copies issued (and, in order, consumed)
    bool bad = false;
    // what the launch asks for besides the step itself (uniform)
    const bool resid = (a.flags & F_RESID) != 0;
    const bool mon = (a.flags & (F_RESID | F_MON)) != 0;
    const bool save_u = (a.flags & F_SAVE_U) != 0;
    const bool want_u = mon || save_u;
    const bool store_sigma = (a.flags & F_STORE_SIGMA) != 0;
    const bool sr = std::is_same<T, __nv_bfloat16>::value && (a.flags & F_SR) != 0;
    const long long PL = ctl.plane;

    auto issue = [&](uint32_t off, int x0, int row) {  // issuing thread (TI) only
        mbar_expect_tx(bar_at(off), TX);
        if constexpr (ODD) {
            const int x = row * nx + x0 - HP;  // (the host keeps planes below 2^31 elements)
            tma_load_3d(slots + off, &tmap, bar_at(off), x - (x & (HP - 1)), 0, 0);
        } else {
            tma_load_3d(slots + off, &tmap, bar_at(off), x0 - HP, row, 0);
        }
    };
    // the slot after the one at `off`
    auto next_slot = [&](uint32_t off) -> uint32_t { return off == (K - 1) * SLOT ? 0u : off + SLOT; };
    uint32_t issued_end = 0;  // issuing thread: one past the index of the last copy issued

    for (int item = blockIdx.x; item < ctl.n_items && !bad && !halted; item += gridDim.x) {
        const MarchItem it = ctl.items[item];
        const int x0 = it.x0, y0 = it.y0, y1 = it.y1, sw = STRIP == kFull ? CW : it.w;
        const int rbase = y0 - 2;                 // first source row of this item
        const int rlast = y1 + 1;                 // last source row
        const uint32_t L0 = nload;                // load index of row rbase
        const bool left_edge = (x0 == 0), right_edge = (x0 + sw == nx);
        // first own column (relative to x0).  Threads beyond a narrower strip repeat its last pair and
        // store nothing; with an odd width the last pair's second column is the halo column
        const int col0 = STRIP == kFull ? 2 * t : min(2 * t, ODD ? (sw - 1) & ~1 : sw - 2);
        const bool own0 = STRIP == kFull || 2 * t < sw, own1 = STRIP == kFull || 2 * t + 1 < sw;
        const bool last_pair = STRIP == kFull ? t == NT - 1 : col0 + 2 == sw;

        // index of the copy holding source row r, its slot, and the wait for it
        auto idx_of = [&](int r) -> uint32_t { return L0 + (uint32_t)(r - rbase); };
        auto slot_off = [&](int r) -> uint32_t { return (idx_of(r) % K) * SLOT; };
        // offset of column x0 - HP of row r inside the slots, given its slot
        auto row_at = [&](uint32_t off, int r) -> uint32_t {
            return ODD ? off + ((uint32_t)(r * nx + x0) & (HP - 1)) * (uint32_t)sizeof(T) : off;
        };
        auto wait_row = [&](int r) -> bool {
            const uint32_t i = idx_of(r);
            return mbar_wait(bar_at((i % K) * SLOT), (i / K) & 1u, ctl.max_wait_ns);
        };
        // periodic wrap: the edge strips' halo columns x0-2, x0-1 (left) or x0+sw, x0+sw+1 (right)
        // come from the other end of the row; threads 0..17 (left) and 32..49 (right) each own
        // one (direction, column) value, loaded two rows before it is patched into its slot
        const bool patcher = (left_edge && t < 18) || (right_edge && t >= 32 && t < 50);
        const int pi = left_edge && t < 18 ? (t >> 1) : ((t - 32) >> 1);             // direction
        const int pc = left_edge && t < 18 ? (nx - 2 + (t & 1)) : ((t - 32) & 1);     // global column
        const int ps = left_edge && t < 18 ? (HP - 2 + (t & 1)) : (HP + sw + ((t - 32) & 1));  // slot column
        auto patch_load = [&](int r) -> T {
            return (r >= 0 && r < ny && r <= rlast) ? a.pin[9 * ctl.base + (long long)pi * PL + (long long)r * nx + pc] : T(0);
        };
        auto patch_store = [&](int r, T v) {
            if (r >= 0 && r < ny && r <= rlast) reinterpret_cast<T*>(slots + row_at(slot_off(r), r))[pi * SW + ps] = v;
        };
        // GPBC brackets: six lanes of the second warp (the first has the halo columns' moments) take one
        // (boundary column, direction) each and evaluate source row r from the
        // slots, which hold the column's raw stored populations (the strip's own edge column, or
        // the halo image of the other end, patched before)
        const bool gpbc_edge = BND == 1 && (left_edge || right_edge) && a.gcol != nullptr;  // CTA-uniform
        const int sl = t - 32;
        const bool shifter = gpbc_edge && sl >= 0 && sl < 6;
        auto shift_row = [&](int r) {
            if (r < 0 || r >= ny || r > rlast) return;
            const int c = sl / 3, j = sl - 3 * (sl / 3);
            const int i = c == 1 ? (j == 0 ? 1 : (j == 1 ? 5 : 8)) : (j == 0 ? 3 : (j == 1 ? 6 : 7));
            const int bcol = c == 1 ? (right_edge ? sw - 1 : -1) : (left_edge ? 0 : sw);
            const T* sb = reinterpret_cast<const T*>(slots + row_at(slot_off(r), r)) + HP + bcol;
            C e[9], mR, mx, my;
#pragma unroll
            for (int k = 0; k < 9; ++k) e[k] = (C)Store<T>::cvt(sb[k * SW]);
            moments<C>(e, mR, mx, my);
            s_shift[BND == 1 ? (r & 7) : 0][c][j] = gpbc_shift_core<C>(i, mR, mx, my, s_delta[c]);
        };
        // The end-crossing corrections (Sec. II B) of one column's populations in row r: the slots hold the raw
        // periodic images, so every population that crosses an end gets its shift where it is pulled.
        // Populations entering x = 0 move with c_x = +1 and leave the column x = nx-1 (END 1: directions
        // 1, 5, 8 from source rows r, r-1, r+1); those entering x = nx-1 move with c_x = -1 and leave
        // x = 0 (END 0: directions 3, 6, 7).  get(i), set(i, v): the column's population of direction i.
        auto cross = [&](auto end, int r, auto get, auto set) {
            constexpr int E = decltype(end)::value, i0 = E ? 1 : 3, i1 = E ? 5 : 6, i2 = E ? 8 : 7;
            auto add_shift = [&](int i, C core) {
                C v = get(i);
                gpbc_add<C>(v, i, core);
                set(i, v);
            };
            add_shift(i0, s_shift[BND == 1 ? (r & 7) : 0][E][0]);
            if (r > 0) add_shift(i1, s_shift[BND == 1 ? ((r - 1) & 7) : 0][E][1]);
            if (r < ny - 1) add_shift(i2, s_shift[BND == 1 ? ((r + 1) & 7) : 0][E][2]);
        };
        using End0 = std::integral_constant<int, 0>;
        using End1 = std::integral_constant<int, 1>;
        // pulled populations of one node (col, r) from the slots (col relative to x0, -1 or CW too):
        // direction i comes from source row r - cy_i, column col - cx_i.  om, o0, op: slot offsets of
        // the source rows r-1, r, r+1
        auto pull_one = [&](int col, int r, uint32_t om, uint32_t o0, uint32_t op, C (&d)[9]) {
            const T* sm = reinterpret_cast<const T*>(slots + row_at(om, r - 1)) + HP + col;
            const T* s0 = reinterpret_cast<const T*>(slots + row_at(o0, r)) + HP + col;
            const T* sp = reinterpret_cast<const T*>(slots + row_at(op, r + 1)) + HP + col;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const bool wall = (cy(i) == 1 && r == 0) || (cy(i) == -1 && r == ny - 1);
                const T* sr = cy(i) == 1 ? sm : (cy(i) == -1 ? sp : s0);
                d[i] = (C)Store<T>::cvt(wall ? s0[opp(i) * SW] : sr[i * SW - cx(i)]);
            }
            if constexpr (BND == 1) {
                if (gpbc_edge) {  // (a halo column beyond an end is the column at the other end)
                    auto get = [&](int i) -> C { return d[i]; };
                    auto set = [&](int i, C v) { d[i] = v; };
                    if (col < 0 && left_edge) cross(End0(), r, get, set);
                    if (col >= sw && right_edge) cross(End1(), r, get, set);
                }
            }
            if constexpr (BND >= 1) {
                if (r == ny - 1 && a.chan[0].moving) zou_he_top<C>(d, a.chan[0].u_wall);
            }
        };
        // the same for the thread's two columns
        auto pull_pair = [&](int r, uint32_t om, uint32_t o0, uint32_t op, P2 (&d)[9]) {
            const T* sm = reinterpret_cast<const T*>(slots + row_at(om, r - 1)) + HP + col0;
            const T* s0 = reinterpret_cast<const T*>(slots + row_at(o0, r)) + HP + col0;
            const T* sp = reinterpret_cast<const T*>(slots + row_at(op, r + 1)) + HP + col0;
            auto even_pair = [&](const T* p) -> P2 {  // (columns of even index: one access where rows are aligned)
                if constexpr (ODD) return slot_pair_odd<T>(p);
                else return slot_pair(p);
            };
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const T* sr = cy(i) == 1 ? sm : (cy(i) == -1 ? sp : s0);
                d[i] = cx(i) == 0 ? even_pair(sr + i * SW) : slot_pair_odd<T>(sr + i * SW - cx(i));
            }
            if (r == 0 || r == ny - 1) {  // bounce-back at the wall (uniform over the CTA)
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    if (cy(i) != 0 && (cy(i) == 1 ? r == 0 : r == ny - 1)) d[i] = even_pair(s0 + opp(i) * SW);
            }
            if constexpr (BND == 1) {
                if (gpbc_edge) {  // the channel's first column is a pair's first; its last a pair's second, at an odd
                                  // strip width (kOdd) its first
                    auto get0 = [&](int i) -> C { return lo(d[i]); };
                    auto set0 = [&](int i, C v) { d[i] = p2(v, hi(d[i])); };
                    auto get1 = [&](int i) -> C { return hi(d[i]); };
                    auto set1 = [&](int i, C v) { d[i] = p2(lo(d[i]), v); };
                    if (left_edge && col0 == 0) cross(End1(), r, get0, set0);
                    if (right_edge && col0 + 2 == sw) cross(End0(), r, get1, set1);
                    if (ODD && right_edge && col0 + 1 == sw) {  // (its second is the halo column, the other end)
                        cross(End0(), r, get0, set0);
                        cross(End1(), r, get1, set1);
                    }
                }
            }
            if (BND >= 1 && r == ny - 1 && a.chan[0].moving) {
                C e0[9], e1[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    e0[i] = lo(d[i]);
                    e1[i] = hi(d[i]);
                }
                zou_he_top<C>(e0, a.chan[0].u_wall);
                zou_he_top<C>(e1, a.chan[0].u_wall);
#pragma unroll
                for (int i = 0; i < 9; ++i) d[i] = p2(e0[i], e1[i]);
            }
        };
        // moments and gradient velocities of row r's own columns.  om, o0, op: slots of rows r-1, r, r+1
        auto moments_row = [&](int r, uint32_t om, uint32_t o0, uint32_t op, P2 (&d)[9], P2& dR, P2& jx, P2& jy, P2& ux,
                               P2& uy) {
            if (r < 0 || r >= ny) return;
            pull_pair(r, om, o0, op, d);
            gradient_velocity(d, q.hgx, dR, jx, jy, ux, uy);
            if constexpr (SHUFFLE) {
                if (t == 31) edge[4 * (r & 3) + 1] = make_float2(hi(ux), hi(uy));
                if (t == 32) edge[4 * (r & 3) + 2] = make_float2(lo(ux), lo(uy));
                if (r == ny - 3) *reinterpret_cast<float4*>(uwall + 2 * col0) = make_float4(lo(ux), lo(uy), hi(ux), hi(uy));
            } else {
                *reinterpret_cast<float4*>(ring(r, col0)) = make_float4(lo(ux), lo(uy), hi(ux), hi(uy));
            }
        };
        // gradient velocities of the two halo columns of row r: one lane per column
        auto halo_node = [&](int r, int col, uint32_t om, uint32_t o0, uint32_t op) {
            C dh[9], hR, hx, hy, hux, huy;
            pull_one(col, r, om, o0, op, dh);
            gradient_velocity<C>(dh, P.gx, hR, hx, hy, hux, huy);
            if constexpr (SHUFFLE) edge[4 * (r & 3) + (col < 0 ? 0 : 3)] = make_float2(hux, huy);
            else *reinterpret_cast<float2*>(ring(r, col)) = make_float2(hux, huy);
        };
        // the own columns' velocities of row r, two rows from a wall
        auto wall_pair = [&](int r, P2& ux, P2& uy) {
            const float4 v = *reinterpret_cast<const float4*>(SHUFFLE ? uwall + 2 * col0 : ring(r, col0));
            ux = p2(v.x, v.z);
            uy = p2(v.y, v.w);
        };

        // ---- prologue: copies of rows rbase .. rbase+K-1; rows rbase .. rbase+5 waited and patched;
        // moments of rows y0-1, y0 (and of row 2 when the item starts at the bottom wall: the
        // one-sided difference of row 0 needs it)
        if (t == TI) {
            fence_proxy_async();
            for (int r = rbase; r < rbase + K && r <= rlast; ++r) {
                issue(slot_off(r), x0, r);
                issued_end = idx_of(r) + 1;
            }
        }
        nload = L0 + (uint32_t)(rlast - rbase + 1);
        // residual partials (F_RESID / F_MON) of this thread's columns, in the arithmetic type (a
        // few hundred rows at most); the block reduction below runs in double
        P2 r_du2 = p2(0.f), r_u2 = p2(0.f), r_ux = p2(0.f);
        C r_umax2 = C(0);
        // populations and moments of the row that collides and of the next one: the row loop is
        // written out for two rows, with the two sets changing places
        P2 dA[9], dB[9];
        P2 dRa, jxa, jya, dRb, jxb, jyb;
        P2 us_x = p2(0.f), us_y = p2(0.f), u0_x, u0_y, un_x = p2(0.f), un_y = p2(0.f);  // rows y-1, y, y+1
        bool ok = true;
        for (int r = rbase; r <= rbase + 5 && r <= rlast; ++r) ok &= wait_row(r);
        if (!ok) s_bad = 1;
        T pv_a = T(0), pv_b = T(0);
        if (patcher && ok) {  // patch only slots whose copies this thread saw land
            for (int r = rbase; r <= rbase + 5; ++r) patch_store(r, patch_load(r));
            pv_a = patch_load(y0 + 4);
            pv_b = patch_load(y0 + 5);
        }
        __syncthreads();
        if (s_bad) { bad = true; break; }
        if (gpbc_edge) {  // brackets of the rows waited and patched so far (CTA-uniform branch)
            if (shifter)
                for (int r = rbase; r <= rbase + 5; ++r) shift_row(r);
            __syncthreads();
        }
        {
            P2 a0, a1, a2, a3, a4;
            moments_row(y0 - 1, slot_off(y0 - 2), slot_off(y0 - 1), slot_off(y0), dA, a0, a1, a2, us_x, us_y);
            if (y0 == 0) {
                moments_row(2, slot_off(1), slot_off(2), slot_off(3), dA, a0, a1, a2, a3, a4);
                if constexpr (SHUFFLE)
                    *reinterpret_cast<float4*>(uwall + 2 * col0) = make_float4(lo(a3), lo(a4), hi(a3), hi(a4));
            }
        }
        moments_row(y0, slot_off(y0 - 1), slot_off(y0), slot_off(y0 + 1), dA, dRa, jxa, jya, u0_x, u0_y);
        if (t < 2) halo_node(y0, t == 0 ? -1 : sw, slot_off(y0 - 1), slot_off(y0), slot_off(y0 + 1));
        // offsets of this item's fields from its first row's first own column
        const long long ubase = ctl.base + (long long)y0 * nx + x0, ibase = ubase + col0;
        // address of the thread's columns in row y of a field: `o` / `vo` rows into the item.  FP32: a
        // CTA-uniform pointer and a 32-bit offset; BF16: per-thread 64-bit pointers (each the faster
        // one for its kernel: FP32 4096 x 4096 253 against 268 us, BF16 8192 x 2048 228 against 223)
        auto field_at = [&](auto* f, long long o, uint32_t vo) {
            using E = std::remove_pointer_t<decltype(f)>;
            if constexpr (OFF32)
                return reinterpret_cast<E*>(reinterpret_cast<uintptr_t>(f + ubase) + (vo + (uint32_t)col0) * (uint32_t)sizeof(E));
            else
                return f + ibase + o;
        };
        // the thread's own columns of a field: one access for both, or (ODD) one each
        auto ld = [&](const C* p) -> P2 {
            if constexpr (ODD) return p2(p[0], own1 ? p[1] : 0.f);
            else return load_pair(p);
        };
        auto st = [&](C* p, P2 v) {
            if constexpr (ODD) {
                if (own0) p[0] = lo(v);
                if (own1) p[1] = hi(v);
            } else if (own0) {
                store_pair(p, v);
            }
        };
        auto st_pop = [&](T* p, P2 v) {
            if constexpr (ODD) {
                if (own0) Store<T>::st(p, lo(v));
                if (own1) Store<T>::st(p + 1, hi(v));
            } else if (own0) {
                store_pop_pair(p, v);
            }
        };
        auto ld_phi = [&](const double* p) -> double2 {
            if constexpr (ODD) return make_double2(p[0], own1 ? p[1] : 0.0);
            else return *reinterpret_cast<const double2*>(p);
        };
        // the stored flow-induced density, loaded two rows ahead of its use
        const C* drow = a.drho + ibase;
        P2 drho_next, drho_next2 = p2(0.f);
        drho_next = ld(drow);
        if (y0 + 1 < y1) drho_next2 = ld(drow + nx);
        // relaxation-time extensions with a fluidity memory: the node's fluidity (FP64), one row ahead
        const bool fluid = SCHEME == 3 && P.tau_f > C(0);  // CTA-uniform
        const double* phrow = a.phi + ibase;
        double2 phi_nxt = make_double2(0.0, 0.0);
        if (fluid) phi_nxt = ld_phi(phrow);
        // on residual steps the saved velocity of each row is prefetched the same way, and one
        // thread brings the delta rho and saved-velocity rows into L2 four rows before their
        // register loads (a residual step reads 16 B more per node than a plain one, and the
        // two-rows-ahead register pipeline alone covers about one row of DRAM latency)
        const C* upx = a.uprev + ctl.base + ibase;
        auto prefetch_rows = [&](int r) {  // thread TP, residual steps, rows of this item only
            if (r < y1) {
                // (whole 16-byte pieces: at an odd width the row's first and last ones are left out)
                const long long o = (long long)r * nx + x0;
                const int lead = ODD ? (int)((4 - (o & 3)) & 3) : 0;
                const uint32_t bytes = (uint32_t)max(0, (sw - lead) / 4) * 16u;
                if (bytes) {
                    prefetch_l2(a.drho + ctl.base + o + lead, bytes);
                    prefetch_l2(a.uprev + 2 * ctl.base + o + lead, bytes);
                    prefetch_l2(a.uprev + 2 * ctl.base + PL + o + lead, bytes);
                }
            }
        };
        P2 upx_next = p2(0.f), upy_next = p2(0.f), upx_next2 = p2(0.f), upy_next2 = p2(0.f);
        if (resid) {
            if (t == TP)
                for (int r = y0 + 2; r < y0 + 6; ++r) prefetch_rows(r);
            upx_next = ld(upx);
            upy_next = ld(upx + PL);
            if (y0 + 1 < y1) {
                upx_next2 = ld(upx + nx);
                upy_next2 = ld(upx + PL + nx);
            }
        }
        __syncthreads();
        if (t == TI) {
            fence_proxy_async();
            for (int r = rbase + K; r < rbase + K + 2 && r <= rlast; ++r) {
                issue(slot_off(r), x0, r);
                issued_end = idx_of(r) + 1;
            }
        }

        long long o = 0;  // offset of row y from the item's first row
        uint32_t vo = 0;  // the same in 32 bits (the host keeps an item's rows below 2^30 elements)
        uint32_t o0 = slot_off(y0), o1 = slot_off(y0 + 1), o2 = slot_off(y0 + 2);  // slots of rows y, y+1, y+2
        uint32_t par2 = (idx_of(y0 + 2) / K) & 1u;                                  // and row y+2's phase
        // one row; false: a wait gave up.  EVEN: the first of two rows
        auto row = [&](const int y, const bool even, P2 (&dcur)[9], P2& dRc, P2& jxc, P2& jyc, P2 (&dnext)[9], P2& dRn, P2& jxn,
                       P2& jyn) -> bool {
            // 1. moments of row y+1 (its own populations are the next row's collision input);
            //    edge strips patch row y+4, which the moments of iteration y+2 read first
            //    edge strips' halo columns: rows y+1 and y+2 are taken in one pass every other row
            if (!mbar_wait(bar_at(o2), par2, ctl.max_wait_ns)) s_bad = 1;  // (y + 2 <= rlast)
            const uint32_t o3 = next_slot(o2);
            const uint32_t par3 = o3 == 0 ? par2 ^ 1u : par2;
            if (patcher && y + 4 <= rlast) {
                if (!wait_row(y + 4)) s_bad = 1;
                else patch_store(y + 4, pv_a);
                pv_a = pv_b;
                pv_b = patch_load(y + 6);
            }
            P2 so_xx = p2(0.f), so_xy = p2(0.f), so_yy = p2(0.f);
            auto carried_stress = [&] {  // of row y
                const C* s3 = a.sig3 + 2 * ctl.base + ibase + o;
                so_xx = ld(s3);
                so_xy = ld(s3 + PL);
                so_yy = ld(s3 + 2 * PL);
            };
            // ahead of the barrier (FP32 4096 x 4096: 334 us, 357 at its use); with the fluidity, whose registers leave no
            // room for it, at its use (2048 x 1024, 16 steps: 1070 us, 1091 here)
            if constexpr (SMODE == 1 && SCHEME != 3) carried_stress();
            moments_row(y + 1, o0, o1, o2, dnext, dRn, jxn, jyn, un_x, un_y);
            // (an end strip with pressure-driven ends: one row, the brackets of row y+3 come too late for two)
            if (!HALO2 || gpbc_edge ? t < 2 : (even && t < 4)) {
                const bool second = t >= 2 && y + 2 < y1;
                if (second && !mbar_wait(bar_at(o3), par3, ctl.max_wait_ns)) s_bad = 1;
                const int r = y + 1 + (t >> 1);
                if ((t < 2 || second) && r < ny)
                    halo_node(r, (t & 1) == 0 ? -1 : sw, second ? o1 : o0, second ? o2 : o1, second ? o3 : o2);
            }
            const P2 drho_prev = drho_next, upx_cur = upx_next, upy_cur = upy_next;
            drho_next = drho_next2;
            if (y + 2 < y1) drho_next2 = ld(field_at(a.drho + 2LL * nx, o, vo));
            double2 phi_cur = phi_nxt;
            if (fluid && y + 1 < y1) phi_nxt = ld_phi(phrow + o + nx);
            if (resid) {
                if (t == TP) prefetch_rows(y + 6);
                upx_next = upx_next2;
                upy_next = upy_next2;
                if (y + 2 < y1) {
                    upx_next2 = ld(upx + o + 2 * nx);
                    upy_next2 = ld(upx + PL + o + 2 * nx);
                }
            }
            __syncthreads();
            if (s_bad) return false;
            // 2. refill the slot of row y (no longer read) with row y+K
            if (t == TI && y + K <= rlast) {
                fence_proxy_async();
                issue(o0, x0, y + K);
                issued_end = idx_of(y + K) + 1;
            }
            // brackets of row y+4: its copy was waited and its halo patched by the patchers before the barrier
            // above (so the wait here returns at once); the first pull that reads it is that of row
            // y+3, two barriers later
            if (shifter && y + 4 <= rlast) {
                (void)wait_row(y + 4);
                shift_row(y + 4);
            }
            // 3. collision of row y, both nodes together, then the row's stores
            {
                // the neighbouring columns' velocities: from the neighbouring lanes (across a warp's
                // border from shared memory), or from the ring
                float2 uw, ue;
                if constexpr (SHUFFLE) {
                    const float2 bw = edge[4 * (y & 3) + wid];
                    const float2 be = edge[4 * (y & 3) + (STRIP == kFull ? 2 + wid : (last_pair ? 3 : 2))];
                    uw = make_float2(__shfl_up_sync(0xffffffffu, hi(u0_x), 1), __shfl_up_sync(0xffffffffu, hi(u0_y), 1));
                    ue = make_float2(__shfl_down_sync(0xffffffffu, lo(u0_x), 1), __shfl_down_sync(0xffffffffu, lo(u0_y), 1));
                    if (lane == 0) uw = bw;
                    if (lane == 31 || (STRIP != kFull && last_pair)) ue = be;
                } else {
                    uw = *reinterpret_cast<const float2*>(ring(y, col0 - 1));
                    ue = *reinterpret_cast<const float2*>(ring(y, col0 + 2));
                }
                const P2 Kx = p2(__fsub_rn(hi(u0_x), uw.x), __fsub_rn(ue.x, lo(u0_x)));
                const P2 Kc = p2(__fsub_rn(hi(u0_y), uw.y), __fsub_rn(ue.y, lo(u0_y)));
                P2 By, Ey;
                if (y == 0) {
                    P2 x2, y2;
                    wall_pair(2, x2, y2);
                    By = wall_difference_first(u0_x, un_x, x2);
                    Ey = wall_difference_first(u0_y, un_y, y2);
                } else if (y == ny - 1) {
                    P2 x2, y2;
                    wall_pair(y - 2, x2, y2);
                    By = wall_difference_last(u0_x, us_x, x2);
                    Ey = wall_difference_last(u0_y, us_y, y2);
                } else {
                    By = sub(un_x, us_x);
                    Ey = sub(un_y, us_y);
                }
                if constexpr (SMODE == 1 && SCHEME == 3) carried_stress();
                PairState s;
                P2 om = q.om, nom = q.nom, k2 = q.k2;
                if constexpr (SCHEME == 1) {
                    s = constitutive_gn(P, q, Kx, By, Kc, Ey, dRc, jxc, jyc, &om);
                    nom = mul(om, p2(-1.f));
                    k2 = fma(p2(-0.5f), om, p2(1.f));
                } else {
                    P2 tau_M = p2(0.f);
                    if constexpr (SCHEME == 3) {
                        double2 phi_new;
                        const C t0 = relaxation_time_ext<C>(P, 0.5f * lo(Kx), 0.5f * lo(By), 0.5f * lo(Kc), 0.5f * lo(Ey),
                                                            lo(dRc), lo(drho_prev), phi_cur.x, &phi_new.x);
                        const C t1 = relaxation_time_ext<C>(P, 0.5f * hi(Kx), 0.5f * hi(By), 0.5f * hi(Kc), 0.5f * hi(Ey),
                                                            hi(dRc), hi(drho_prev), phi_cur.y, &phi_new.y);
                        tau_M = p2(t0, t1);
                        if (!FIELDS && fluid) {
                            double* ph = a.phi + ibase + o;
                            if constexpr (ODD) {
                                if (own0) ph[0] = phi_new.x;
                                if (own1) ph[1] = phi_new.y;
                            } else if (own0) {
                                *reinterpret_cast<double2*>(ph) = phi_new;
                            }
                        }
                    }
                    s = constitutive<SMODE, BND == 1, SCHEME == 3>(q, Kx, By, Kc, Ey, dRc, jxc, jyc, drho_prev, so_xx, so_xy,
                                                                   so_yy, tau_M);
                }
                const P2 rho_h = sub(add(p2(1.f), s.dReq), s.drho);
                if constexpr (FIELDS) {
                    const P2 ih = rcp(rho_h), urx = mul(jxc, ih), ury = mul(jyc, ih);
                    const long long node = (long long)y * nx + x0 + col0;
                    if (own0) store_fields<C>(a, node, lo(urx), lo(ury), lo(s.sxx), lo(s.syy), lo(s.sxy), lo(rho_h));
                    if (own1) store_fields<C>(a, node + 1, hi(urx), hi(ury), hi(s.sxx), hi(s.syy), hi(s.sxy), hi(rho_h));
                }
                {  // velocity_ok of both nodes: |u| <= guard without a division (false for NaN)
                    const P2 j2 = fma(jyc, jyc, mul(jxc, jxc)), g2 = mul(mul(p2(a.guard * a.guard), rho_h), rho_h);
                    vbad |= (own0 & !(lo(j2) <= lo(g2))) | (own1 & !(hi(j2) <= hi(g2)));
                }
                if constexpr (!FIELDS) {
                P2 D[9];
                collide<SCHEME != 0>(q, s, dcur, D, om, nom, k2);
                T* po = a.pout + 8 * ctl.base;
                if (sr) {
                    // store_node's draws and rounding, both nodes' values in one store; whether all are finite
                    // (its exception) is asked once: BF16 4096 x 4096 258 us, 368 value by value
                    if constexpr (!F32) {
                        const uint32_t node = (uint32_t)((long long)y * nx + x0 + col0);
                        P2 nan = p2(0.f);
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            D[i] = add(dcur[i], D[i]);
                            nan = fma(D[i], p2(0.f), nan);  // (NaN from an infinity or a NaN)
                        }
                        if (!(lo(nan) + hi(nan) == 0.f)) {
                            C n0[9], n1[9];
#pragma unroll
                            for (int i = 0; i < 9; ++i) {
                                n0[i] = lo(D[i]);
                                n1[i] = hi(D[i]);
                            }
                            if (own0) store_node<T, C>(field_at(po, o, vo), PL, n0, true, a.sr_key, node);
                            if (own1) store_node<T, C>(field_at(po, o, vo) + 1, PL, n1, true, a.sr_key, node + 1);
                        } else {
                            uint32_t h0 = 0, h1 = 0;
#pragma unroll
                            for (int i = 0; i < 9; ++i) {
                                if ((i & 1) == 0) {
                                    h0 = mix32(a.sr_key ^ (node * 5u + (uint32_t)(i >> 1)));
                                    h1 = mix32(a.sr_key ^ ((node + 1) * 5u + (uint32_t)(i >> 1)));
                                }
                                const uint32_t b0 = __float_as_uint(lo(D[i])) + ((i & 1) ? h0 >> 16 : h0 & 0xffffu);
                                const uint32_t b1 = __float_as_uint(hi(D[i])) + ((i & 1) ? h1 >> 16 : h1 & 0xffffu);
                                T* p = field_at(po + i * PL, o, vo);
                                if constexpr (ODD) {
                                    if (own0) p[0] = __ushort_as_bfloat16((unsigned short)(b0 >> 16));
                                    if (own1) p[1] = __ushort_as_bfloat16((unsigned short)(b1 >> 16));
                                } else if (own0) {
                                    *reinterpret_cast<uint32_t*>(p) = __byte_perm(b0, b1, 0x7632);
                                }
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i) st_pop(field_at(po + i * PL, o, vo), add(dcur[i], D[i]));
                }
                st(field_at(a.drho, o, vo), s.drho);
                if (SMODE == 1) {
                    C* s3 = a.sig3 + 2 * ctl.base + ibase + o;
                    st(s3, s.sxx);
                    st(s3 + PL, s.sxy);
                    st(s3 + 2 * PL, s.syy);
                }
                if (store_sigma) {  // (the zz plane holds 0 from lb_create on)
                    C* s4 = a.sig4 + 3 * ctl.base;
                    st(field_at(s4, o, vo), s.sxx);
                    st(field_at(s4 + PL, o, vo), s.syy);
                    st(field_at(s4 + 3 * PL, o, vo), s.sxy);
                }
                if (want_u) {
                    const P2 ih = rcp(rho_h);
                    const P2 urx = mul(jxc, ih), ury = mul(jyc, ih);
                    if (mon) {
                        // (threads and halves without a column of their own add zeros, whatever they hold)
                        auto mask = [&](P2 v) { return STRIP == kFull ? v : p2(own0 ? lo(v) : 0.f, own1 ? hi(v) : 0.f); };
                        const P2 u2 = mask(fma(ury, ury, mul(urx, urx)));
                        if (resid) {
                            const P2 dx_ = sub(urx, upx_cur), dy_ = sub(ury, upy_cur);
                            r_du2 = add(r_du2, mask(fma(dy_, dy_, mul(dx_, dx_))));
                        }
                        r_u2 = add(r_u2, u2);
                        r_ux = add(r_ux, mask(urx));
                        r_umax2 = fmaxf(r_umax2, fmaxf(lo(u2), hi(u2)));
                    }
                    if (save_u) {
                        C* up_ = a.uprev + ctl.base + ibase + o;
                        st(up_, urx);
                        st(up_ + PL, ury);
                    }
                }
                }  // not the fields pass
            }
            us_x = u0_x;
            us_y = u0_y;
            u0_x = un_x;
            u0_y = un_y;
            o0 = o1;
            o1 = o2;
            o2 = o3;
            par2 = par3;
            o += nx;
            vo += (uint32_t)nx;
            return true;
        };
        if constexpr (!UNROLL2) {
#pragma unroll 1
            for (int y = y0; y < y1; ++y) {
                if (!row(y, ((y - y0) & 1) == 0, dA, dRa, jxa, jya, dB, dRb, jxb, jyb)) { bad = true; break; }
#pragma unroll
                for (int i = 0; i < 9; ++i) dA[i] = dB[i];
                dRa = dRb;
                jxa = jxb;
                jya = jyb;
            }
        } else {
            for (int y = y0; y < y1; y += 2) {
                if (!row(y, true, dA, dRa, jxa, jya, dB, dRb, jxb, jyb)) { bad = true; break; }
                if (y + 1 >= y1) break;
                if (!row(y + 1, false, dB, dRb, jxb, jyb, dA, dRa, jxa, jya)) { bad = true; break; }
            }
        }
        __syncthreads();  // every slot read of this item is done before the next item's copies
        if (!bad && mon) {
            // block reduction of (sum du^2, sum u^2, sum u_x, max u^2) into this item's partials: few FP64 operations
            // (a butterfly over four doubles, and the last block's over every item by one warp, made a
            // monitored step of 1024 x 1024 nodes 7 us longer: 16 of them, with the force set and the monitor read, 684
            // -> 565 us)
            double v0 = resid ? (double)lo(r_du2) + (double)hi(r_du2) : 0.0;
            const double v1 = (double)lo(r_u2) + (double)hi(r_u2), v2 = (double)lo(r_ux) + (double)hi(r_ux);
            warp_sum3(v0, v1, v2, lane);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) r_umax2 = fmaxf(r_umax2, __shfl_xor_sync(0xffffffffu, r_umax2, o));
            double* red = reinterpret_cast<double*>(uwall);  // (free now)
            if ((lane & 7) == 0 && lane < 24) red[4 * wid + (lane >> 3)] = v0;
            if (lane == 0) red[4 * wid + 3] = (double)r_umax2;
            __syncthreads();
            if (t < 4) a.partials[4 * (long long)item + t] = t < 3 ? red[t] + red[4 + t] : max_pos(red[3], red[7]);
            __syncthreads();
        }
    }

    if (vbad) atomicOr(a.status, 1);
    if (bad) {
        // record the timeout and drain this CTA's own copies before leaving: a slot is refilled
        // only after every thread's wait on its previous copy succeeded, so the last copy issued
        // into each slot is the only one that can still be in flight (bounded by kMarchDrainNs)
        if (t == TI) {
            atomicOr(ctl.timeout_flag, 2);
            for (uint32_t k = issued_end > (uint32_t)K ? issued_end - K : 0u; k < issued_end; ++k)
                mbar_wait(bar_at((k % K) * SLOT), (k / K) & 1u, kMarchDrainNs);
        }
        __syncthreads();
    }
    if (ctl.done_count != nullptr) {  // the last CTA to get here: status mirror and monitor
        __shared__ bool s_last;
        __syncthreads();
        if (t == 0) {
            __threadfence();  // this CTA's partials and status bits before its count
            s_last = atomicAdd(ctl.done_count, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (s_last) {
            __threadfence();
            const int st = *(volatile const int*)a.status;
            if (ctl.mon != nullptr)
                monitor_reduce<NT / 32>(a.partials, 0, ctl.n_items, st, ctl.mon, nx, ctl.state_index, ctl.with_residual, t, true,
                                        reinterpret_cast<double*>(uwall));
            if (t == 0) {
                if (ctl.status_host != nullptr) *(volatile int*)ctl.status_host = st;
                *ctl.done_count = 0u;
            }
        }
    }
}

}  // namespace lbk

namespace lbk {
// How the kernel is shaped, and what it measured (us per step; FP32 at 4096 x 4096 / 1024 x 1024, BF16
// at 8192 x 2048 / 1024 x 1024; one column per thread in scalar FP32 before: 274 / 24.8 and 222 / 24.8).
// Two columns per thread as packed FP32 take the instructions per node from 468 to 268 (FP32) and from
// 393 to 268 (BF16); what is left is bound by HBM in FP32 at sizes beyond L2 (0.9 of the copy
// bandwidth) and by the latency of dependent instructions elsewhere: a packed operation holds its
// warp for about four cycles, and 160 registers leave 12 warps per SM.
//  - six CTAs of two warps per SM.  Eight (128 registers) spill, or pull the populations twice: BF16
//    218 / 22.9 against 215 / 20.8.
//  - seven row slots: with the halo columns of two rows taken together (which waits one row
//    further ahead) six slots leave too little in flight for HBM (FP32 293 / 20.8 against 253 / 22.4).
//    Seven fit six CTAs in FP32 without the ring of velocity rows, hence the warp shuffles; BF16 has
//    the room and keeps the ring (215 / 20.8 against 223 / 20.8 with shuffles).
//  - the row loop written out for two rows, so that no register moves between them: BF16 230 -> 215;
//    with pressure-driven ends FP32 is faster one row at a time (2048 x 1000: 51.6 against 53.0), BF16
//    (4096 x 4096) is not (275 against 255).  A loop of its own for the end strips, the other strips running that
//    of the periodic channels, was slower than either (53.2 and 274: two bodies share an SM).
constexpr int kMarchK = 7;  // shared-memory row slots

template <typename T, typename C, int SMODE, int BND = 0, int SCHEME = 0, bool FIELDS = false, int STRIP = 0>
cudaError_t launch_step_march(const CUtensorMap& map, const StepArgs<T, C>& a, const MarchCtl& ctl, int grid,
                              cudaStream_t s) {
    constexpr int K = kMarchK;
    auto k = k_step_march<T, C, SMODE, kMarchW, K, BND, SCHEME, FIELDS, STRIP>;
    const size_t smem = march_smem_bytes<T, C, kMarchW, K, STRIP == kOdd>();
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    return launch_dependent(ctl.dependent, k, grid, kMarchW / 2, smem, s, map, a, ctl);
}

template <typename T, typename C, int SMODE, int BND = 0, int SCHEME = 0, int STRIP = 0>
cudaError_t march_occupancy(int* blocks_per_sm) {
    constexpr int K = kMarchK;
    auto k = k_step_march<T, C, SMODE, kMarchW, K, BND, SCHEME, false, STRIP>;
    const size_t smem = march_smem_bytes<T, C, kMarchW, K, STRIP == kOdd>();
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, kMarchW / 2, smem);
}
}  // namespace lbk
// Every variant (stress mode, boundary, scheme) of the kernel for storage type T; X(T, SMODE, BND, SCHEME).
#define LB_MARCH_VARIANTS(X, T)                                                          \
    X(T, 0, 0, 0) X(T, 1, 0, 0) X(T, 0, 1, 0) X(T, 1, 1, 0) X(T, 0, 2, 0) X(T, 1, 2, 0) \
    X(T, 0, 0, 1) X(T, 0, 0, 3) X(T, 1, 0, 3)
// Its instantiations for steps (with the occupancy query) and for the fields pass.
#define LB_MARCH_STEP(PREFIX, T, SMODE, BND, SCHEME, STRIP)                                                                  \
    PREFIX template cudaError_t launch_step_march<T, float, SMODE, BND, SCHEME, false, STRIP>(                              \
        const CUtensorMap&, const StepArgs<T, float>&, const MarchCtl&, int, cudaStream_t);                                \
    PREFIX template cudaError_t march_occupancy<T, float, SMODE, BND, SCHEME, STRIP>(int*);
#define LB_MARCH_FIELDS(PREFIX, T, SMODE, BND, SCHEME, STRIP)                                                                \
    PREFIX template cudaError_t launch_step_march<T, float, SMODE, BND, SCHEME, true, STRIP>(                               \
        const CUtensorMap&, const StepArgs<T, float>&, const MarchCtl&, int, cudaStream_t);
