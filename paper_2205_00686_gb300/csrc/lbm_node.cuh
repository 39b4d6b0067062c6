// Arithmetic of one node of the two-dimensional step, shared by the kernels
// that advance it (k_step sweeps strips of rows, k_tile steps small domains).
// Every operation is written with its rounding fixed (a product is never
// contracted into a later sum unless fma says so), so that a node's result
// does not depend on the kernel, the tile or the compiler's scheduling: the
// kernels agree bit for bit, and a domain gets the same populations alone, in
// a batch or in another tile.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {

__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// Two-lane arithmetic.  In float it maps to Blackwell's paired FP32
// instructions (one FADD2 / FMUL2 / FFMA2 does the work of two), each lane
// rounded as the scalar operation; in double it is componentwise.  Subtraction
// is a fused multiply-add with -1, which is exact in the product.
template <class R> struct Vec2;
template <> struct Vec2<float> { typedef float2 T; };
template <> struct Vec2<double> { typedef double2 T; };
__device__ __forceinline__ float2 pr(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 pr(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 padd(double2 a, double2 b) { return pr(radd(a.x, b.x), radd(a.y, b.y)); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 pmul(double2 a, double2 b) { return pr(rmul(a.x, b.x), rmul(a.y, b.y)); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c) {
    return pr(rfma(a.x, b.x, c.x), rfma(a.y, b.y, c.y));
}
// c - a b
__device__ __forceinline__ float2 pnfma(float2 a, float2 b, float2 c) {
    return __ffma2_rn(a, make_float2(-b.x, -b.y), c);
}
__device__ __forceinline__ double2 pnfma(double2 a, double2 b, double2 c) {
    return pr(rfma(-a.x, b.x, c.x), rfma(-a.y, b.y, c.y));
}
__device__ __forceinline__ float2 psub(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}
__device__ __forceinline__ double2 psub(double2 a, double2 b) { return pr(rsub(a.x, b.x), rsub(a.y, b.y)); }

// psi^2 and E = T (dp/dT)_rho / (12 rho c_v) of one node, with D1 = 1 - b rho
// and D2 = 1 + 2 b rho - b^2 rho^2 = 2 - D1^2 over one common reciprocal:
//   p = rho (Rg T D2 - a h^2 rho D1) / (D1 D2)
//   T (dp/dT)_rho = rho (Rg T D2 + a k h sqrt(T/Tc) rho D1) / (D1 D2)
// (T / sqrt(T/Tc) = Tc sqrt(T/Tc), so no second reciprocal, and E needs none of
// rho).  One square root and one reciprocal, 18 other operations with sqrt(a)
// taken into h.  (For a < 0, which needs R < 0, p and the constants that meet it
// carry the other sign.)
template <class R>
__device__ __forceinline__ void eos_node(const Phys<R>& P, R rho, R T, R* psi2, R* E) {
    const R st = f_sqrt(rmul(T, P.inv_Tc));
    const R h = rfma(-P.k_sa, st, P.k1_sa);      // sqrt(a) h
    const R d1 = rfma(-P.b, rho, R(1));
    const R d2 = rfma(-d1, d1, R(2));
    const R rc = f_rcp(rmul(d1, d2));
    const R u = rmul(rmul(P.Rg, T), d2), w = rmul(rho, d1);
    const R p = rmul(rmul(rho, rc), rfma(-rmul(h, h), w, u));
    *psi2 = rmul(P.two_over_G, rfma(rho, P.m_third, p));
    *E = rmul(rmul(P.inv_12cv, rc), rfma(rmul(rmul(P.k_sa, st), h), w, u));
}

// What the later stages take of a node's populations and EOS
template <class R>
struct Node {
    R rho, rhod;      // density and its deviation from the storage reference
    R T, Td;          // temperature and its deviation
    R jx, jy;
    R m7, m8;         // stress moments (unit rates)
    R ir;             // 1 / rho
    R C, iC;          // rho c_v and its reciprocal as the blend takes it
    R E;              // T (dp/dT)_rho / (12 rho c_v)
    R q2, psi;        // psi^2 and psi
};

// 1/(rho c_v) of the weighted streaming.  FP64 forms it from 1/rho (three
// FP64 operations fewer); FP32 with the hardware reciprocal of rho c_v, which
// spares carrying one more value from stage to stage.
__device__ __forceinline__ float blend_iC(float C, float) { return f_rcp(C); }
__device__ __forceinline__ double blend_iC(double, double iC) { return iC; }

// T - T_ref: sum of the deviations of g
template <class R>
__device__ __forceinline__ R sum5(const R* g) {
    const typename Vec2<R>::T p = padd(pr(g[1], g[2]), pr(g[3], g[4]));
    return radd(radd(g[0], p.x), p.y);
}

// rho - rho_ref: sum of the deviations of f, in the order of node_fields
template <class R>
__device__ __forceinline__ R sum9(const R* f) {
    const typename Vec2<R>::T sA = padd(pr(f[1], f[2]), pr(f[3], f[4]));
    const typename Vec2<R>::T sB = padd(pr(f[5], f[6]), pr(f[7], f[8]));
    return radd(radd(f[0], radd(sA.x, sA.y)), radd(sB.x, sB.y));
}

// moments, EOS and psi of a node from its (deviation) populations
template <class R>
__device__ __forceinline__ void node_fields(const Phys<R>& P, R rho_ref, R T_ref, const R* f,
                                            const R* g, Node<R>& n) {
    typedef typename Vec2<R>::T R2;
    // pair sums and differences of (f1, f2) & (f3, f4) and (f5, f6) & (f7, f8)
    const R2 sA = padd(pr(f[1], f[2]), pr(f[3], f[4]));   // (f1 + f3, f2 + f4)
    const R2 dA = psub(pr(f[1], f[2]), pr(f[3], f[4]));   // (f1 - f3, f2 - f4)
    const R2 sB = padd(pr(f[5], f[6]), pr(f[7], f[8]));   // (f5 + f7, f6 + f8)
    const R2 dB = psub(pr(f[5], f[6]), pr(f[7], f[8]));   // (f5 - f7, f6 - f8)
    n.rhod = radd(radd(f[0], radd(sA.x, sA.y)), radd(sB.x, sB.y));
    n.rho = radd(n.rhod, rho_ref);
    n.ir = f_rcp(n.rho);
    n.Td = sum5(g);
    n.T = radd(n.Td, T_ref);
    n.jx = radd(dA.x, rsub(dB.x, dB.y));    // (f1 - f3) + (f5 - f7) - (f6 - f8)
    n.jy = radd(dA.y, radd(dB.x, dB.y));    // (f2 - f4) + (f5 - f7) + (f6 - f8)
    n.m7 = rsub(sA.x, sA.y);
    n.m8 = rsub(sB.x, sB.y);
    eos_node(P, n.rho, n.T, &n.q2, &n.E);
    n.psi = f_sqrt(n.q2);
    n.C = rmul(n.rho, P.cv);
    n.iC = rmul(n.ir, P.inv_cv);
}

// ghost-layer psi of a wall (Section 3.3): rho_ghost = rho(layer 2) +
// tan(pi/2 - theta) |rho(x+1, layer 1) - rho(x-1, layer 1)|, at the temperature
// of the fluid node next to it
template <class R>
__device__ __forceinline__ R ghost_psi(const Phys<R>& P, R rho_far, R rho_p, R rho_m, R cot, R Tg,
                                       int* err) {
    const R rg = rfma(cot, rabs(rsub(rho_p, rho_m)), rho_far);
    R q2, E;
    eos_node(P, rg, Tg, &q2, &E);
    if (!(q2 >= R(0))) *err |= (q2 != q2) ? ERR_NONFINITE : ERR_PSI;
    return f_sqrt(q2);
}

// force stencil of Eq. 9 with varpi(1) = 1/3, varpi(2) = 1/12, both components
// at once: 12 s = 4 (pE - pW, pN - pS) + (dA + dB, dA - dB)
template <class R>
__device__ __forceinline__ typename Vec2<R>::T force_stencil(R pW, R pE, R pSW, R pS, R pSE, R pNW,
                                                             R pN, R pNE) {
    const R dA = rsub(pNE, pSW), dB = rsub(pSE, pNW);
    return pfma(psub(pr(pE, pN), pr(pW, pS)), pr(R(4), R(4)), pr(radd(dA, dB), rsub(dA, dB)));
}

// F = F_m + F_b (Section 4.3)
template <class R>
__device__ __forceinline__ typename Vec2<R>::T force_of(const Phys<R>& P, typename Vec2<R>::T s12,
                                                        R psi, R rho, R rho_ave) {
    const R gp = rmul(P.negG_12, psi);
    typename Vec2<R>::T F = pmul(pr(gp, gp), s12);
    // (without gravity FP64 spares its two operations)
    if (sizeof(R) == 4 || P.gravity != R(0)) F.y = rfma(-P.gravity, rsub(rho, rho_ave), F.y);
    return F;
}

// u = (j + F/2) / rho (Eq. 11)
template <class R, class R2>
__device__ __forceinline__ R2 velocity(R2 F, R2 j, R ir) {
    return pmul(pfma(F, pr(R(0.5), R(0.5)), j), pr(ir, ir));
}

// D2Q9 collision at unit rates (s_e = s_eps = s_q = 1: those moments leave the
// collision at m^eq + F/2), so f* = M^{-1} m* needs of f only rho, j and the
// stress moments m_7, m_8 (Eqs. 5, 7, 8).  With K = rho u.u + u.F and
// |12 s|^2 of the force stencil,
//   f*_0          = what the others leave of rho (4/9 rho - 2/3 K + ...)
//   axis part     = 1/9 rho + 1/12 K + u_ax |12 s|^2, +- m*_7/4, +- (j + F)/3
//   diagonal part = 1/36 rho + 1/12 K + u_dg |12 s|^2, +- m*_8/4,
//                   +- ((j + F)_x +- (j + F)_y)/12
// With f*_0 as the remainder and the float 1/12 rounded down, so that 2/3 + 4/12
// is 1, mass and momentum are kept to the rounding of the populations (each
// weight rounded by itself adds 3e-8 of them every step in FP32).  In FP64, where
// that is 1e-16, it is formed from its own weight as the oracle does (fields of
// 1999 x 1501 after 10 steps 2.3e-15 off the oracle's, as remainder 2.8e-15).
// With rho u = j + F/2 the products with u come in two groups: u_a (j + 3/2 F)_a
// sums to K, and u_a w_b with w = s_p/4 rho u + (1 - s_p/2)/2 F is what the
// stresses take.  rhod: deviation of rho from the storage reference (f is stored
// as deviations).
template <class R, class R2>
__device__ __forceinline__ void collide9_unit(const Phys<R>& P, R rhod, R2 j, R m7, R m8,
                                              R2 u, R2 F, R2 s12, R* f, int stride) {
    const R2 v = pfma(F, pr(R(1.5), R(1.5)), j);
    const R2 w = pfma(F, pr(P.u_w, P.u_w), pmul(j, pr(P.u_d, P.u_d)));
    const R K = rfma(u.x, v.x, rmul(u.y, v.y));
    const R S = rfma(s12.x, s12.x, rmul(s12.y, s12.y));
    const R b7 = rfma(P.u_m, m7, rfma(u.x, w.x, -rmul(u.y, w.y)));
    const R b8 = rfma(P.u_m, m8, rmul(R(0.5), rfma(u.x, w.y, rmul(u.y, w.x))));
    const R K12 = rmul(K, R(1.0 / 12.0));
    const R2 cc = pfma(pr(rhod, rhod), pr(R(1.0 / 9.0), R(1.0 / 36.0)),
                       pfma(pr(S, S), pr(P.u_ax, P.u_dg), pr(K12, K12)));
    const R2 js = padd(j, F);
    // axis directions: (1, 2) = (ax + b7, ax - b7) + js/3, (3, 4) the same
    // minus js/3; diagonals: (5, 8) = (dg + b8, dg - b8) + (jx + jy, jx - jy)/12,
    // (7, 6) the same minus that
    const R2 cb = pr(radd(cc.x, b7), rsub(cc.x, b7)), db = pr(radd(cc.y, b8), rsub(cc.y, b8));
    const R2 sd = pr(radd(js.x, js.y), rsub(js.x, js.y));
    const R w12 = sizeof(R) == 4 ? R(0x1.555554p-4) : R(1.0 / 12.0);
    const R2 t3 = pr(R(1.0 / 3.0), R(1.0 / 3.0)), t12 = pr(w12, w12);
    const R2 f12 = pfma(js, t3, cb), f58 = pfma(sd, t12, db);
    const R2 f34 = pnfma(js, t3, cb), f76 = pnfma(sd, t12, db);
    f[0] = sizeof(R) == 4 ? rfma(R(-4), radd(cc.x, cc.y), rhod)
                          : rfma(R(4.0 / 9.0), rhod, rfma(R(-2.0 / 3.0), K, rmul(P.u_0, S)));
    f[1 * stride] = f12.x;
    f[2 * stride] = f12.y;
    f[3 * stride] = f34.x;
    f[4 * stride] = f34.y;
    f[5 * stride] = f58.x;
    f[6 * stride] = f76.y;
    f[7 * stride] = f76.x;
    f[8 * stride] = f58.y;
}

// D2Q9 collision at general rates: f* = f + M^{-1} (m* - m), m* - m =
// -S (m - m^eq) + (I - S/2) F (Eqs. 5, 7, 8), with M^{-1} = M^T diag(1/9, 1/36,
// 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4)
template <class R, class R2>
__device__ __forceinline__ void collide9(const Phys<R>& P, R rho, R rhod, const R* f, R2 u, R2 F,
                                         R2 s12, R* out, int stride) {
    const R ux = u.x, uy = u.y, Fx = F.x, Fy = F.y;
    const R rux = rmul(rho, ux), ruy = rmul(rho, uy);
    const R ruu = rfma(rux, ux, rmul(ruy, uy));
    const R s13 = radd(f[1], f[3]), s24 = radd(f[2], f[4]);
    const R s57 = radd(f[5], f[7]), s68 = radd(f[6], f[8]);
    const R s14 = radd(s13, s24), s58 = radd(s57, s68);
    // non-equilibrium parts m - m^eq of the moments of Eq. 7 (deviation
    // storage shifts m_e by -2 rho_ref, m_eps by rho_ref)
    const R ne1 = rfma(R(-3), ruu, rfma(R(2), rsub(radd(s58, rhod), f[0]), -rfma(R(2), f[0], s14)));
    const R ne2 = rfma(R(3), ruu, rsub(radd(rfma(R(4), f[0], rmul(R(-2), s14)), s58), rhod));
    const R d13 = rsub(f[1], f[3]), d24 = rsub(f[2], f[4]);
    const R d58 = rsub(f[5], f[7]), d68 = rsub(f[6], f[8]);
    const R ne4 = radd(rfma(R(-2), d13, rsub(d58, d68)), rux);
    const R ne6 = radd(rfma(R(-2), d24, radd(d58, d68)), ruy);
    const R ne7 = rsub(rsub(s13, s24), rfma(rux, ux, -rmul(ruy, uy)));
    const R ne8 = rfma(-rux, uy, rsub(s57, s68));
    // Li forcing (Eq. 8); |F_m|^2 / psi^2 = G^2 |sum varpi psi c|^2
    const R uF = rfma(ux, Fx, rmul(uy, Fy));
    const R Fm2 = rmul(rmul(P.negG_12, P.negG_12), rfma(s12.x, s12.x, rmul(s12.y, s12.y)));
    const R F1 = rfma(R(6), uF, rmul(P.sig_e, Fm2));
    const R F2 = rfma(R(-6), uF, -rmul(P.sig_eps, Fm2));
    const R F7 = rmul(R(2), rfma(ux, Fx, -rmul(uy, Fy)));
    const R F8 = rfma(ux, Fy, rmul(uy, Fx));
    // for j the change is exactly F because rho u = j + F/2
    const R a1m = rmul(rfma(P.hs_e, F1, -rmul(P.s_e, ne1)), R(1.0 / 36.0));
    const R a2m = rmul(rfma(P.hs_eps, F2, -rmul(P.s_eps, ne2)), R(1.0 / 36.0));
    const R a3 = rmul(Fx, R(1.0 / 6.0)), a5 = rmul(Fy, R(1.0 / 6.0));
    const R a4 = rmul(rfma(P.s_q, ne4, rmul(P.hs_q, Fx)), R(-1.0 / 12.0));
    const R a6 = rmul(rfma(P.s_q, ne6, rmul(P.hs_q, Fy)), R(-1.0 / 12.0));
    const R a7 = rmul(rfma(P.hs_p, F7, -rmul(P.s_p, ne7)), R(0.25));
    const R a8 = rmul(rfma(P.hs_p, F8, -rmul(P.s_p, ne8)), R(0.25));
    const R cax = rfma(R(-2), a2m, -a1m);   // common to the axis directions
    const R cdg = rfma(R(2), a1m, a2m);     // common to the diagonals
    const R ex = rfma(R(-2), a4, a3), ey = rfma(R(-2), a6, a5);
    const R dx = radd(a3, a4), dy = radd(a5, a6);
    out[0] = rfma(R(4), rsub(a2m, a1m), f[0]);
    out[1 * stride] = radd(radd(radd(f[1], cax), ex), a7);
    out[2 * stride] = rsub(radd(radd(f[2], cax), ey), a7);
    out[3 * stride] = radd(rsub(radd(f[3], cax), ex), a7);
    out[4 * stride] = rsub(rsub(radd(f[4], cax), ey), a7);
    out[5 * stride] = radd(radd(radd(radd(f[5], cdg), dx), dy), a8);
    out[6 * stride] = rsub(radd(rsub(radd(f[6], cdg), dx), dy), a8);
    out[7 * stride] = radd(rsub(rsub(radd(f[7], cdg), dx), dy), a8);
    out[8 * stride] = rsub(rsub(radd(radd(f[8], cdg), dx), dy), a8);
}

// isotropic central difference, 12 (1/c_s^2) sum_i w_i c_i . u(x + c_i)
template <class R, class R2>
__device__ __forceinline__ R div12_of(R2 uW, R2 uE, R2 uS0, R2 uS1, R2 uS2, R2 uN0, R2 uN1, R2 uN2) {
    const R ax = radd(rsub(uE.x, uW.x), rsub(uN1.y, uS1.y));
    const R dx = radd(rsub(uN2.x, uN0.x), rsub(uS2.x, uS0.x));
    const R dy = radd(rsub(uN2.y, uS2.y), rsub(uN0.y, uS0.y));
    return rfma(R(4), ax, radd(dx, dy));
}

// Thermal stage of a node: P^n (Eq. 20) and the D2Q5 MRT collision (Eqs. 39,
// 40, 47) of its (deviation) populations g.
//   P^n = Q / (rho c_v) = -[u.grad T + T (dp/dT)_rho div u / (rho c_v)] with
//   c_s^2 grad T = -varsigma_1 (m_1, m_2) (Eqs. 49-50, m^eq = 0);
//   S = w^ rho c_v (dt/2) d_t^2 T with d_t^2 T ~ P^n - P^{n-1} (Eq. 24), so
//   Q + S = rho c_v (P^n + (P^n - P^{n-1}) / 2).
template <bool UNIT, class R, class R2>
__device__ __forceinline__ R thermal5(const Phys<R>& P, const R* g, R Td, R C, R E, R2 u, R div12,
                                      R Pp, bool first, R* gs) {
    // (m_1, m_2) = (g1 - g3, g2 - g4)
    const R2 m12 = psub(pr(g[1], g[2]), pr(g[3], g[4]));
    const R Pn = rfma(P.vs1_cs2h, rfma(u.x, m12.x, rmul(u.y, m12.y)), -rmul(E, div12));
    const R dP = first ? Pn : rfma(R(0.5), rsub(Pn, Pp), Pn);
    const R2 h12 = pmul(pr(P.h_m, P.h_m), m12);     // (1 - varsigma_1)/2 m
    if (UNIT) {
        // varsigma_3 = varsigma_4 = 1: m3* = w_dot (T + Q + S), m4* = 0
        const R TQ = rfma(C, dP, Td);
        const R a = rmul(P.w5_1, TQ);
        // FP32: what the others leave of T (see collide9_unit)
        gs[0] = sizeof(R) == 4 ? rfma(R(-4), a, TQ) : rmul(P.w5_0, TQ);
        const R2 g12 = padd(pr(a, a), h12), g34 = psub(pr(a, a), h12);
        gs[1] = g12.x;
        gs[2] = g12.y;
        gs[3] = g34.x;
        gs[4] = g34.y;
    } else {
        const R Qs = rmul(C, dP);
        const R s13 = radd(g[1], g[3]), s24 = radd(g[2], g[4]);
        const R m3d = radd(s13, s24), m4 = rsub(s13, s24);
        const R m0s = radd(Td, Qs);
        const R m3s = rfma(P.w_dot, Qs, rfma(-P.vs3, rfma(-P.w_dot, Td, m3d), m3d));
        const R m4s = rmul(P.one_m_vs4, m4);
        const R a = rmul(R(0.25), radd(m3s, m4s)), b = rmul(R(0.25), rsub(m3s, m4s));
        gs[0] = rsub(m0s, m3s);
        gs[1] = radd(a, h12.x);
        gs[2] = radd(b, h12.y);
        gs[3] = rsub(a, h12.x);
        gs[4] = rsub(b, h12.y);
    }
    return Pn;
}

// weighted streaming (Eq. 39): g + (A - g) / (rho c_v)
template <class R>
__device__ __forceinline__ R blend(R g, R A, R iC) { return rfma(rsub(A, g), iC, g); }

}  // namespace lbm
