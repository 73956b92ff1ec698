// lb_pair.cuh -- the per-node arithmetic of lb_device.cuh on two nodes at once, in packed FP32.
//
// sm_103a executes add, mul and fma on a pair of FP32 values held in one 64-bit register
// (add/sub/mul/fma.rn.f32x2, each lane rounded to nearest as the scalar instruction).  The FP32 rate is
// the scalar one -- measured 39.0e12 scalar and 40.0e12 paired FMA lanes/s on the whole part -- but a
// pair takes one issue slot instead of two, and the step kernels are bound by instruction issue
// (70 % of the slots taken, "not selected" the largest stall), not by the FP32 units.
//
// Every expression names its operations (no contraction is left to the compiler) and rounds in the
// order in which the compiler rounds the scalar expressions of lb_device.cuh, so a kernel that works on
// pairs gives the bits of one that works node by node; the tests compare the two.  Exact scalings
// by powers of two are moved where they save an operation.
#pragma once

#include "lb_device.cuh"

namespace lbk {

// Two FP32 values, lo in the low half.
struct P2 {
    unsigned long long v;
};

__device__ __forceinline__ P2 p2(float lo, float hi) {
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ P2 p2(float both) { return p2(both, both); }
__device__ __forceinline__ float lo(P2 a) {
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return x;
}
__device__ __forceinline__ float hi(P2 a) {
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return y;
}
__device__ __forceinline__ P2 add(P2 a, P2 b) {
    P2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 sub(P2 a, P2 b) {
    P2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 mul(P2 a, P2 b) {
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 fma(P2 a, P2 b, P2 c) {
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// reciprocal and square root: the scalar routines of Arith<float>, lane by lane
__device__ __forceinline__ P2 rcp(P2 a) {
    return p2(Arith<float>::div(1.f, lo(a)), Arith<float>::div(1.f, hi(a)));
}
__device__ __forceinline__ P2 root(P2 a) { return p2(Arith<float>::sqrt(lo(a)), Arith<float>::sqrt(hi(a))); }

// Channel constants of the pair arithmetic, broadcast to both lanes.
struct PairConst {
    P2 om, nom, k1, nk1, k1x2, nk1x2, k2, gx, hgx, G, tau, igc, cD, kdr;
};
__device__ __forceinline__ PairConst pair_const(const ChanParams<float>& P) {
    PairConst q;
    q.om = p2(P.omega);
    q.nom = p2(-P.omega);
    q.k1 = p2(P.k1);
    q.nk1 = p2(-P.k1);
    q.k1x2 = p2(2.f * P.k1);
    q.nk1x2 = p2(-2.f * P.k1);
    q.k2 = p2(P.k2);
    q.gx = p2(P.gx);
    q.hgx = p2(0.5f * P.gx);
    q.G = p2(P.G);
    q.tau = p2(P.tau);
    q.igc = p2(P.inv_gc);
    q.cD = p2(P.cD);
    q.kdr = p2(P.kdr);
    return q;
}

// gradient_velocity (Eq. rhoj and j / R0) of two nodes
__device__ __forceinline__ void gradient_velocity(const P2 (&d)[9], P2 hgx, P2& dR, P2& jx, P2& jy, P2& ux, P2& uy) {
    dR = add(add(add(add(d[0], d[1]), add(d[2], d[3])), add(add(d[4], d[5]), add(d[6], d[7]))), d[8]);
    jx = add(add(add(sub(d[1], d[3]), sub(d[5], d[6])), sub(d[8], d[7])), hgx);
    jy = sub(add(sub(d[2], d[4]), add(d[5], d[6])), add(d[7], d[8]));
    const P2 inv = rcp(add(p2(1.f), dR));
    ux = mul(jx, inv);
    uy = mul(jy, inv);
}

// One-sided difference of the first (2 d/dy = -3 u0 + 4 u1 - u2) and last (3 u0 - 4 u1 + u2) row.
__device__ __forceinline__ P2 wall_difference_first(P2 u0, P2 u1, P2 u2) {
    return sub(fma(p2(4.f), u1, mul(p2(-3.f), u0)), u2);
}
__device__ __forceinline__ P2 wall_difference_last(P2 u0, P2 u1, P2 u2) {
    return add(fma(p2(3.f), u0, mul(p2(-4.f), u1)), u2);
}

struct PairState {
    P2 sxx, sxy, syy;  // polymer stress
    P2 Bxx, Bxy;       // traceless Sigma^nN
    P2 drho, S, dReq, ux, uy;
};

// Twice the shear-rate invariant's argument, D, and its root: D = kappa + kappa^T from the doubled
// three-point differences Kx = 2 d_x u_x, By = 2 d_y u_x, Kc = 2 d_x u_y, Ey = 2 d_y u_y.
__device__ __forceinline__ P2 shear_rate(P2 Kx, P2 W, P2 Dxy, P2 Ey) {
    return root(mul(p2(0.5f), fma(Ey, Ey, fma(Kx, Kx, mul(W, Dxy)))));
}

// constitutive (lb_device.cuh) of two nodes.  KDR: the flow-induced density may be switched off (kdr
// of the channel, pressure-driven ends); otherwise it is on.  TAUM: tau_M comes in.
template <int SMODE, bool KDR, bool TAUM>
__device__ __forceinline__ PairState constitutive(const PairConst& q, P2 Kx, P2 By, P2 Kc, P2 Ey, P2 dR, P2 jx, P2 jy,
                                                  P2 drho_prev, P2 so_xx, P2 so_xy, P2 so_yy, P2 tau_M) {
    PairState r;
    const P2 half = p2(0.5f), one = p2(1.f);
    const P2 W = add(By, Kc);
    const P2 Dxy = mul(half, W);
    if constexpr (!TAUM) tau_M = mul(q.tau, rcp(fma(mul(q.tau, shear_rate(Kx, W, Dxy, Ey)), q.igc, one)));
    P2 al = tau_M, b1, b2, b3;
    if constexpr (SMODE == 0) {
        const P2 gt = mul(q.G, al);
        b1 = mul(gt, Kx);
        b2 = mul(gt, Dxy);
        b3 = mul(gt, Ey);
    } else {
        al = mul(tau_M, rcp(add(tau_M, one)));
        b1 = mul(al, fma(q.G, Kx, so_xx));
        b2 = mul(al, fma(q.G, Dxy, so_xy));
        b3 = mul(al, fma(q.G, Ey, so_yy));
    }
    // convected_solve; 2 alpha kappa_ab = alpha x doubled difference, halved right-hand sides hb
    const P2 nal = mul(al, p2(-1.f));
    const P2 A = fma(nal, Kx, one), E = fma(nal, Ey, one);
    const P2 Pp = fma(mul(al, p2(-0.5f)), add(Kx, Ey), one);
    const P2 al2B = mul(mul(al, al), By), al2K = mul(mul(al, al), Kc);
    const P2 q4 = mul(al2B, Kc), nq2 = mul(p2(-0.5f), q4);
    const P2 AE = mul(A, E);
    const P2 id = rcp(mul(Pp, sub(AE, q4)));
    const P2 aB = mul(al, By), aK = mul(al, Kc);
    const P2 hb1 = mul(half, b1), hb3 = mul(half, b3);
    const P2 aKE = mul(aK, E), aBA = mul(aB, A);
    r.sxy = mul(fma(aBA, hb3, fma(aKE, hb1, mul(AE, b2))), id);
    r.sxx = mul(fma(mul(al2B, By), hb3, fma(mul(aB, E), b2, mul(fma(Pp, E, nq2), b1))), id);
    r.syy = mul(fma(fma(A, Pp, nq2), b3, fma(mul(al2K, Kc), hb1, mul(mul(aK, A), b2))), id);
    const P2 Nxx = fma(q.cD, Kx, r.sxx), Nxy = fma(q.cD, Dxy, r.sxy), Nyy = fma(q.cD, Ey, r.syy);
    r.drho = mul(p2(-1.5f), add(Nxx, Nyy));
    if constexpr (KDR) {
        r.drho = mul(q.kdr, r.drho);
        r.S = sub(r.drho, mul(q.kdr, drho_prev));
    } else {
        r.S = sub(r.drho, drho_prev);
    }
    r.Bxx = mul(half, sub(Nxx, Nyy));
    r.Bxy = Nxy;
    r.dReq = fma(half, r.S, dR);
    const P2 inv = rcp(add(one, r.dReq));
    r.ux = mul(jx, inv);
    r.uy = mul(jy, inv);
    return r;
}

// constitutive_gn of two nodes (the generalized-Newtonian scheme); *om receives 1/tau_LB.
__device__ __forceinline__ PairState constitutive_gn(const ChanParams<float>& P, const PairConst& q, P2 Kx, P2 By, P2 Kc,
                                                     P2 Ey, P2 dR, P2 jx, P2 jy, P2* om) {
    PairState r;
    const P2 one = p2(1.f), W = add(By, Kc), Dxy = mul(p2(0.5f), W);
    const P2 tau_M = mul(q.tau, rcp(fma(mul(q.tau, shear_rate(Kx, W, Dxy, Ey)), q.igc, one)));
    const P2 gt = mul(q.G, tau_M);
    r.sxx = mul(gt, Kx);
    r.sxy = mul(gt, Dxy);
    r.syy = mul(gt, Ey);
    r.Bxx = r.Bxy = r.drho = r.S = p2(0.f);
    r.dReq = dR;
    const P2 inv = rcp(add(one, dR));
    r.ux = mul(jx, inv);
    r.uy = mul(jy, inv);
    *om = rcp(fma(p2(P.gn_a), tau_M, p2(P.gn_b)));
    return r;
}

// collide_impl of two nodes: D_i with the force density (gx, 0).  om, nom = -om and k2 are the channel's
// or (GEN) the node's own.  GEN also rounds Y_yy on its own, as the scalar routine's general form does.
template <bool GEN>
__device__ __forceinline__ void collide(const PairConst& q, const PairState& s, const P2 (&d)[9], P2 (&D)[9], P2 om,
                                        P2 nom, P2 k2) {
    const P2 ux = s.ux, uy = s.uy, gx = q.gx;
    const P2 w1 = p2(wgt<float>(1)), w5 = p2(wgt<float>(5));
    const P2 w13 = p2(wgt<float>(1) * 3.f), w53 = p2(wgt<float>(5) * 3.f), nw53 = p2(-(wgt<float>(5) * 3.f));
    const P2 c45 = p2(4.5f), nth = p2(-(1.f / 3.f));
    const P2 rq = add(p2(1.f), s.dReq);
    const P2 orq = mul(om, rq);
    const P2 usq = fma(ux, ux, mul(uy, uy));
    const P2 nS = mul(s.S, p2(-1.f));
    const P2 sux = mul(nS, ux), suy = mul(nS, uy);
    const P2 Yxx = fma(add(ux, ux), gx, mul(sux, ux));
    const P2 Yxy = fma(uy, gx, mul(sux, uy));
    const P2 sumY = fma(suy, uy, Yxx);
    const P2 ntr = mul(sumY, nth);
    const P2 xT = fma(sumY, nth, Yxx);
    const P2 yT = GEN ? fma(sumY, nth, mul(suy, uy)) : fma(suy, uy, ntr);
    const P2 Yxy2 = add(Yxy, Yxy);
    const P2 T5 = add(add(sumY, Yxy2), ntr), T8 = add(sub(sumY, Yxy2), ntr);
    const P2 base = fma(k2, s.S, mul(om, fma(mul(rq, p2(-1.5f)), usq, s.dReq)));
    {
        const P2 oc = mul(orq, ux);
        const P2 XE = fma(q.k1, s.Bxx, fma(c45, fma(oc, ux, mul(k2, xT)), base));
        D[1] = fma(nom, d[1], fma(w13, fma(k2, gx, oc), mul(w1, XE)));
    }
    {
        const P2 oc = mul(orq, uy);
        const P2 XE = fma(q.nk1, s.Bxx, fma(c45, fma(oc, uy, mul(k2, yT)), base));
        D[2] = fma(nom, d[2], fma(w13, oc, mul(w1, XE)));
    }
    {
        const P2 cu = add(ux, uy), oc = mul(orq, cu);
        const P2 E = mul(w5, fma(q.k1x2, s.Bxy, fma(c45, fma(oc, cu, mul(k2, T5)), base)));
        const P2 O = fma(k2, gx, oc);
        D[5] = fma(nom, d[5], fma(w53, O, E));
        D[7] = fma(nom, d[7], fma(nw53, O, E));
    }
    {
        const P2 cu = sub(ux, uy), oc = mul(orq, cu);
        const P2 E = mul(w5, fma(q.nk1x2, s.Bxy, fma(c45, fma(oc, cu, mul(k2, T8)), base)));
        const P2 O = fma(k2, gx, oc);
        D[8] = fma(nom, d[8], fma(w53, O, E));
        D[6] = fma(nom, d[6], fma(nw53, O, E));
    }
    const P2 d57 = sub(D[5], D[7]);
    D[3] = sub(add(add(D[1], d57), sub(D[8], D[6])), gx);
    D[4] = add(add(D[2], d57), sub(D[6], D[8]));
    D[0] = sub(s.S, add(add(add(D[1], D[2]), add(D[3], D[4])), add(add(D[5], D[6]), add(D[7], D[8]))));
}

}  // namespace lbk
