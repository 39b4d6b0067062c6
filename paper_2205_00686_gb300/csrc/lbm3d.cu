// Three-dimensional form of the coupled step: D3Q19 MRT pseudopotential flow
// lattice (d'Humieres moment basis, Li forcing with the sigma term on the
// energy moment) + D3Q7 temperature lattice with the rho c_v-weighted
// streaming of Eq. 39, x and y periodic, z periodic or walls.
//
// Two forms of the step give the same result.  Both start with
//   k3_macro    rho, j, the stress moments, psi, T dp/dT of the state from
//               f(t), g(t), and the density sum for buoyancy
// Then k3_march (below; the default in FP32) does the rest of the step in one
// kernel over z-marching tiles.  The other form (the default in FP64) is two
// more kernels over the nodes plus a one-thread counter update:
//   k3_flow     psi of the 18 neighbours (ghost layer at walls) -> F_m, F,
//               u = (j + F/2)/rho, |F_m|^2/psi^2; D3Q19 collision, f* pushed
//               to its destination (bounce-back at walls)    (Eqs. 5, 9, 11)
//   k3_thermal  div u (neighbour u), grad T (local moments), Q, P^n, S;
//               D3Q7 collision; g*_i blended into the destination's
//               g(t+1) = g + (g* - g)/(rho c_v) (anti-bounce-back at walls),
//               P^n stored                             (Eqs. 20, 24, 39)
//
// Populations are stored as deviations f_i - w_i rho_ref and g_i - w^_i T_ref,
// in blocks of 32 nodes along x: a block holds its 19 (or 7) populations one
// after the other, 32 nodes each (128 bytes in FP32), so all populations of a
// node lie at constant offsets from one address (as planes they need 64-bit
// address arithmetic for each) and a tile row of 32 nodes is one block.
// The other per-node fields are planes [nz][ny][pitch], 64-bit offsets.
//
// At unit rates (s_e = s_eps = s_q = 1 and varsigma_3 = varsigma_4 = 1, the
// paper's setting) the collision needs of f only rho, j and the five stress
// moments (collide19_unit): about 300 operations per node and step instead
// of 770, which is what bounds the FP64 step, and no moment matrices (96^3
// FP64 in the step over nodes: 1080 -> 514 us).
#include <math.h>
#include <string.h>

#include <new>
#include <string>
#include <type_traits>
#include <utility>

#include "lbm.h"
#include "lbm3d.h"
#include "lbm_node.cuh"

namespace lbm {
namespace {

// ---- D3Q19 / D3Q7 tables as constexpr functions (folded after unrolling) --
__host__ __device__ constexpr int qx(int i) {
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
           : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__host__ __device__ constexpr int qy(int i) {
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
           : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
}
__host__ __device__ constexpr int qz(int i) {
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
           : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
}
__host__ __device__ constexpr int qopp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
__host__ __device__ constexpr int qc2(int i) { return qx(i) * qx(i) + qy(i) * qy(i) + qz(i) * qz(i); }
__host__ __device__ constexpr double qw(int i) {
    return qc2(i) == 0 ? 1.0 / 3.0 : (qc2(i) == 1 ? 1.0 / 18.0 : 1.0 / 36.0);
}
// moment k of direction i (d'Humieres et al. 2002 basis), integer valued
__host__ __device__ constexpr int mrow(int k, int i) {
    return k == 0 ? 1
         : k == 1 ? 19 * qc2(i) - 30
         : k == 2 ? (21 * qc2(i) * qc2(i) - 53 * qc2(i) + 24) / 2
         : k == 3 ? qx(i)
         : k == 4 ? (5 * qc2(i) - 9) * qx(i)
         : k == 5 ? qy(i)
         : k == 6 ? (5 * qc2(i) - 9) * qy(i)
         : k == 7 ? qz(i)
         : k == 8 ? (5 * qc2(i) - 9) * qz(i)
         : k == 9 ? 3 * qx(i) * qx(i) - qc2(i)
         : k == 10 ? (3 * qc2(i) - 5) * (3 * qx(i) * qx(i) - qc2(i))
         : k == 11 ? qy(i) * qy(i) - qz(i) * qz(i)
         : k == 12 ? (3 * qc2(i) - 5) * (qy(i) * qy(i) - qz(i) * qz(i))
         : k == 13 ? qx(i) * qy(i)
         : k == 14 ? qy(i) * qz(i)
         : k == 15 ? qx(i) * qz(i)
         : k == 16 ? (qy(i) * qy(i) - qz(i) * qz(i)) * qx(i)
         : k == 17 ? (qz(i) * qz(i) - qx(i) * qx(i)) * qy(i)
                   : (qx(i) * qx(i) - qy(i) * qy(i)) * qz(i);
}
// squared norm of row k (the basis is orthogonal: M^-1 = M^T diag(1/norm))
__host__ __device__ constexpr int mnorm(int k) {
    int s = 0;
    for (int i = 0; i < 19; ++i) s += mrow(k, i) * mrow(k, i);
    return s;
}
// Parity of a moment row under c -> -c: the even rows take the same entry
// for a direction and its opposite, the odd rows opposite entries (and none
// for the rest direction).  Pairs are p = 1..9: directions 2p - 1 and 2p.
__host__ __device__ constexpr bool row_even(int k) {
    for (int p = 1; p <= 9; ++p)
        if (mrow(k, 2 * p - 1) != mrow(k, 2 * p)) return false;
    return true;
}
__host__ __device__ constexpr bool row_odd(int k) {
    if (mrow(k, 0) != 0) return false;
    for (int p = 1; p <= 9; ++p)
        if (mrow(k, 2 * p - 1) != -mrow(k, 2 * p)) return false;
    return true;
}
constexpr bool rows_split() {
    for (int k = 0; k < 19; ++k)
        if (row_even(k) == row_odd(k)) return false;
    for (int p = 1; p <= 9; ++p)
        if (qopp(2 * p - 1) != 2 * p) return false;
    return true;
}
static_assert(rows_split(), "every moment row is even or odd under c -> -c");

// f(integral_constant<int, 0>) ... f(integral_constant<int, N - 1>): the
// index is a constant in every call, whatever the unroller decides
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// m = M f from the pair sums S_p = f_{2p-1} + f_{2p} (even rows) and
// differences D_p = f_{2p-1} - f_{2p} (odd rows): about half the operations
// of the plain product
template <class R>
__device__ __forceinline__ void moments19(const R (&f)[19], R (&m)[19]) {
    R S[10], Dp[10];
    static_for<9>([&](auto pc) {
        constexpr int p = decltype(pc)::value + 1;
        S[p] = f[2 * p - 1] + f[2 * p];
        Dp[p] = f[2 * p - 1] - f[2 * p];
    });
    static_for<19>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        R s = 0;
        if constexpr (mrow(k, 0) != 0) s = R(mrow(k, 0)) * f[0];
        static_for<9>([&](auto pc) {
            constexpr int p = decltype(pc)::value + 1;
            constexpr int c = mrow(k, 2 * p - 1);
            if constexpr (c != 0) s += R(c) * (row_odd(k) ? Dp[p] : S[p]);
        });
        m[k] = s;
    });
}

// f += M^T dm: for each pair the even rows give one term E_p for both
// directions, the odd rows a term O_p of opposite signs
template <class R>
__device__ __forceinline__ void add_inverse19(const R (&dm)[19], R (&f)[19]) {
    R E0 = 0;
    static_for<19>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if constexpr (mrow(k, 0) != 0) E0 += R(mrow(k, 0)) * dm[k];
    });
    f[0] += E0;
    static_for<9>([&](auto pc) {
        constexpr int p = decltype(pc)::value + 1;
        R E = 0, O = 0;
        static_for<19>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            constexpr int c = mrow(k, 2 * p - 1);
            if constexpr (c != 0) {
                if constexpr (row_odd(k)) O += R(c) * dm[k];
                else E += R(c) * dm[k];
            }
        });
        f[2 * p - 1] += E + O;
        f[2 * p] += E - O;
    });
}

// D3Q7: rest, +-x, +-y, +-z
__host__ __device__ constexpr int hx(int i) { return i == 1 ? 1 : (i == 2 ? -1 : 0); }
__host__ __device__ constexpr int hy(int i) { return i == 3 ? 1 : (i == 4 ? -1 : 0); }
__host__ __device__ constexpr int hz(int i) { return i == 5 ? 1 : (i == 6 ? -1 : 0); }

// per-node planes: the fields of the current state (rho as its deviation from
// rho_ref, which keeps the precision of the populations), E = T dp/dT / (12 rho
// c_v), and, for the step over nodes and the read-out, T, u and IC = 1/(rho c_v)
// (k3_flow, once it has read the node's j_x)
enum { Q_RHO = 0, Q_PSI, Q_E, Q_JX, Q_JY, Q_JZ, Q_S, Q_T = Q_S + 5, Q_UX, Q_UY, Q_UZ, Q_N,
       Q_IC = Q_JX };

// Blocks of XB nodes along x: population i of node n at fofs(n) + i XB, gofs(n)
// + i XB (the pitch is a multiple of 32)
constexpr int XB = 32;
__host__ __device__ __forceinline__ size_t fofs(size_t n) { return (n / XB) * (19 * XB) + n % XB; }
__host__ __device__ __forceinline__ size_t gofs(size_t n) { return (n / XB) * (7 * XB) + n % XB; }

struct Dom3 {
    void* f[2];
    void* g[2];
    void* P[2];
    void* aux;
    Ctl* ctl;
    int nx, ny, nz, pitch;
    size_t plane;
    int walls, therm[2];
    double T_edge[2], cot, rho_ref, T_ref, inv_n;
};

template <class R>
struct Lat3 {
    R s_e, s_eps, s_q, s_p;
    R sig_e3;            // (19/2) sigma / (1/s_e - 1/2), the sigma term of e
    R vs3, vs4, w7_0, w7_1, cv, inv_cv, gravity;
    // unit rates: 1 - s_p, a quarter of it, 2 - s_p/2; the sigma term's factors of |12 s|^2 in the
    // axis and diagonal populations; (1 - vs1)/2; vs1 / cs2h
    R c_m, c_m4, c_w, h_ax, h_dg, h_m, vs1_cs2h;
    R rho_ref, T_ref;
    R tw2[2];            // 2 w^_i (T_wall - T_ref) of the bottom and the top
    int frozen_flow, frozen_thermal;
};

template <class R>
Lat3<R> make_lat3(const lbm_params& p, const Dom3& D) {
    Lat3<R> L;
    L.s_e = (R)p.s_e;
    L.s_eps = (R)p.s_eps;
    L.s_q = (R)p.s_q;
    const double s_p = 1.0 / (3.0 * p.nu + 0.5);
    L.s_p = (R)s_p;
    L.sig_e3 = (R)(9.5 * p.sigma / (1.0 / p.s_e - 0.5));
    L.c_m = (R)(1.0 - s_p);
    L.c_m4 = (R)(0.25 * (1.0 - s_p));
    L.c_w = (R)(2.0 - 0.5 * s_p);
    {
        // half the sigma source of e, as a factor of |12 s|^2 = 144 |F_m|^2 / (G psi)^2,
        // times the row entries over the row's norm
        const double h = 0.5 * 9.5 * p.sigma / (1.0 / p.s_e - 0.5) * p.G * p.G / 144.0;
        L.h_ax = (R)(h * mrow(1, 1) / (double)mnorm(1));
        L.h_dg = (R)(h * mrow(1, 7) / (double)mnorm(1));
    }
    L.rho_ref = (R)D.rho_ref;
    L.T_ref = (R)D.T_ref;
    const double cs2h = p.w_dot / 3.0;
    L.vs3 = (R)p.vs3;
    L.vs4 = (R)p.vs4;
    L.w7_0 = (R)(1.0 - p.w_dot);
    L.w7_1 = (R)(p.w_dot / 6.0);
    L.h_m = (R)(0.5 * (1.0 - 1.0 / (p.lambda / cs2h + 0.5)));
    L.vs1_cs2h = (R)(1.0 / (p.lambda / cs2h + 0.5) / cs2h);
    for (int e = 0; e < 2; ++e) L.tw2[e] = (R)(2.0 * (p.w_dot / 6.0) * (D.T_edge[e] - D.T_ref));
    L.cv = (R)p.cv;
    L.inv_cv = (R)(1.0 / p.cv);
    L.gravity = (R)p.gravity;
    L.frozen_flow = p.frozen_flow;
    L.frozen_thermal = p.frozen_thermal;
    return L;
}

// the EOS / interaction constants shared with the two-dimensional kernels
PhysD phys_of(const lbm_params& p) {
    PhysD d;
    memset(&d, 0, sizeof(d));
    d.a = p.a;
    d.b = p.b;
    d.Rg = p.R;
    d.omega = p.omega;
    d.G = p.G;
    d.sigma = p.sigma;
    d.s_e = p.s_e;
    d.s_eps = p.s_eps;
    d.s_q = p.s_q;
    d.s_p = 1.0 / (3.0 * p.nu + 0.5);
    d.cv = p.cv;
    d.w_dot = p.w_dot;
    d.vs1 = 1.0 / (p.lambda / (p.w_dot / 3.0) + 0.5);
    d.vs3 = p.vs3;
    d.vs4 = p.vs4;
    d.gravity = p.gravity;
    d.frozen_flow = p.frozen_flow;
    d.frozen_thermal = p.frozen_thermal;
    return d;
}

// ---- node arithmetic -------------------------------------------------------
// rho - rho_ref, j and the five stress moments (3p_xx, p_ww, p_xy, p_yz, p_xz) of
// a node's populations, from the sums and differences of opposite directions
template <class R>
struct Mom3 {
    R rhod, j[3], st[5];
};

template <bool STRESS, class R>
__device__ __forceinline__ void moments3(const R* f, Mom3<R>& m) {
    typedef typename Vec2<R>::T R2;
    const R2 s12 = padd(pr(f[1], f[3]), pr(f[2], f[4])), d12 = psub(pr(f[1], f[3]), pr(f[2], f[4]));
    const R s3 = f[5] + f[6], d3 = f[5] - f[6];
    const R2 s45 = padd(pr(f[7], f[9]), pr(f[8], f[10])), d45 = psub(pr(f[7], f[9]), pr(f[8], f[10]));
    const R2 s67 = padd(pr(f[11], f[13]), pr(f[12], f[14])), d67 = psub(pr(f[11], f[13]), pr(f[12], f[14]));
    const R2 s89 = padd(pr(f[15], f[17]), pr(f[16], f[18])), d89 = psub(pr(f[15], f[17]), pr(f[16], f[18]));
    const R xy = s45.x + s45.y, xz = s67.x + s67.y, yz = s89.x + s89.y;
    const R yz_ax = s12.y + s3;
    m.rhod = (f[0] + (s12.x + yz_ax)) + ((xy + xz) + yz);
    m.j[0] = d12.x + ((d45.x + d45.y) + (d67.x + d67.y));
    m.j[1] = d12.y + ((d45.x - d45.y) + (d89.x + d89.y));
    m.j[2] = d3 + ((d67.x - d67.y) + (d89.x - d89.y));
    if (STRESS) {
        m.st[0] = R(2) * (s12.x - yz) + ((xy + xz) - yz_ax);
        m.st[1] = (s12.y - s3) + (xy - xz);
        m.st[2] = s45.x - s45.y;
        m.st[3] = s89.x - s89.y;
        m.st[4] = s67.x - s67.y;
    }
}

// D3Q19 collision at unit rates: the moments but rho, j and the stresses leave
// it at m^eq + F/2, so f* = M^{-1} m* closes over rho, j + F, K = rho u.u + u.F
// and the relaxed stresses N = (1 - s_p) m + s_p m^eq + (1 - s_p/2) F:
//   rest      rho less the others (rho/3 - K/2 + h_0 |12 s|^2)
//   axis a    rho/18 + h_ax |12 s|^2 + stress_a +- (j + F)_a / 6
//   diagonal  rho/36 + K/24 + h_dg |12 s|^2 + stress_ab +- N_ab/4
//             +- ((j + F)_a +- (j + F)_b) / 12
// (the pi moments enter the stress parts at -1/2 of their p counterparts'
// equilibrium + F/2).  The rest population is what the others leave of rho and
// 1/6 is rounded down, 1/12 up, so that 2/6 + 8/12 is 1: with each weight
// rounded by itself mass and momentum grow by 3e-8 a step in FP32 (256^3 after
// 100 steps: fields 1.4e-6 off the FP64 ones).  With the products with u grouped
// as below and E without a reciprocal of its own the step has 16 operations fewer
// than with each moment by itself (96^3 FP64 540 -> 514 us).
template <class R>
__device__ __forceinline__ void collide19_unit(const Lat3<R>& L, const Mom3<R>& m, const R* u,
                                               const R* F, R S, R* f) {
    // equilibrium + force as products with u (rho u = j + F/2): g = u_a (rho u + F)_a
    // gives K and m^eq + F/2 of 3p_xx and p_ww (their force rows are twice u_a F_a's),
    // w = s_p rho u + (2 - s_p) F the relaxed stresses
    const R gx = u[0] * (m.j[0] + R(1.5) * F[0]), gy = u[1] * (m.j[1] + R(1.5) * F[1]),
            gz = u[2] * (m.j[2] + R(1.5) * F[2]);
    const R gyz = gy + gz, K = gx + gyz;
    const R pxx = R(2) * gx - gyz, pww = gy - gz;
    const R wx = L.s_p * m.j[0] + L.c_w * F[0], wy = L.s_p * m.j[1] + L.c_w * F[1],
            wz = L.s_p * m.j[2] + L.c_w * F[2];
    const R ty = u[1] * wy, tz = u[2] * wz;
    const R n9 = L.c_m * m.st[0] + (R(2) * (u[0] * wx) - (ty + tz));
    const R n11 = L.c_m * m.st[1] + (ty - tz);
    // N_ab / 4
    const R q13 = L.c_m4 * m.st[2] + R(0.125) * (u[0] * wy + u[1] * wx);
    const R q14 = L.c_m4 * m.st[3] + R(0.125) * (u[1] * wz + u[2] * wy);
    const R q15 = L.c_m4 * m.st[4] + R(0.125) * (u[0] * wz + u[2] * wx);
    // stress parts: N/36 (or N/12) and (m^eq + F/2)/72 (or /24)
    const R p9 = n9 * R(1.0 / 36.0), p11 = n11 * R(1.0 / 12.0);
    const R pa = pxx * R(1.0 / 72.0) + p9, pd = pxx * R(-1.0 / 144.0) + p9;
    const R qa = pww * R(1.0 / 24.0) + p11, qd = pww * R(-1.0 / 48.0) + p11;
    const R ax = m.rhod * R(1.0 / 18.0) + L.h_ax * S;
    const R dg = m.rhod * R(1.0 / 36.0) + (K * R(1.0 / 24.0) + L.h_dg * S);
    const R jx = m.j[0] + F[0], jy = m.j[1] + F[1], jz = m.j[2] + F[2];
    const R a0 = ax + R(2) * pa, a1 = (ax - pa) + qa, a2 = (ax - pa) - qa;
    const R dxy = (dg + pd) + qd, dxz = (dg + pd) - qd, dyz = dg - R(2) * pd;
    const R c6 = sizeof(R) == 4 ? R(0x1.555554p-3) : R(1.0 / 6.0), c12 = R(1.0 / 12.0);
    f[0] = (m.rhod - R(6) * ax) - R(12) * dg;
    f[1] = a0 + c6 * jx;
    f[2] = a0 - c6 * jx;
    f[3] = a1 + c6 * jy;
    f[4] = a1 - c6 * jy;
    f[5] = a2 + c6 * jz;
    f[6] = a2 - c6 * jz;
    const R e7 = dxy + q13, e9 = dxy - q13, e11 = dxz + q15, e13 = dxz - q15;
    const R e15 = dyz + q14, e17 = dyz - q14;
    const R o7 = jx + jy, o9 = jx - jy, o11 = jx + jz, o13 = jx - jz, o15 = jy + jz, o17 = jy - jz;
    f[7] = e7 + c12 * o7;
    f[8] = e7 - c12 * o7;
    f[9] = e9 + c12 * o9;
    f[10] = e9 - c12 * o9;
    f[11] = e11 + c12 * o11;
    f[12] = e11 - c12 * o11;
    f[13] = e13 + c12 * o13;
    f[14] = e13 - c12 * o13;
    f[15] = e15 + c12 * o15;
    f[16] = e15 - c12 * o15;
    f[17] = e17 + c12 * o17;
    f[18] = e17 - c12 * o17;
}

// D3Q19 collision at general rates, in moment space: f* = f + M^T dm with
// dm = (-S (m - m^eq) + (I - S/2) Fbar) / |row|^2 (d'Humieres equilibria:
// w_eps = 3, w_epsj = -11/2, w_xx = -1/2); Fm2 = |F_m|^2 / psi^2
template <class R>
__device__ __forceinline__ void collide19(const Lat3<R>& L, R rho, const R* u, const R* F, R Fm2, R (&f)[19]) {
    R m[19];
    moments19(f, m);
    // deviation storage: m(abs) = m(dev) + rho_ref M w, M w = (1, -11, 3, 0 ...)
    m[0] += L.rho_ref;
    m[1] += R(-11) * L.rho_ref;
    m[2] += R(3) * L.rho_ref;
    const R ux = u[0], uy = u[1], uz = u[2], Fx = F[0], Fy = F[1], Fz = F[2];
    const R uu = ux * ux + uy * uy + uz * uz;
    const R uF = ux * Fx + uy * Fy + uz * Fz;
    R meq[19], Fb[19], sk[19];
    meq[0] = rho;                            Fb[0] = 0;                  sk[0] = 0;
    meq[1] = rho * (R(-11) + R(19) * uu);    Fb[1] = R(38) * uF + L.sig_e3 * Fm2;  sk[1] = L.s_e;
    meq[2] = rho * (R(3) - R(5.5) * uu);     Fb[2] = R(-11) * uF;        sk[2] = L.s_eps;
    meq[3] = rho * ux;                       Fb[3] = Fx;                 sk[3] = 1;
    meq[4] = R(-2.0 / 3.0) * rho * ux;       Fb[4] = R(-2.0 / 3.0) * Fx; sk[4] = L.s_q;
    meq[5] = rho * uy;                       Fb[5] = Fy;                 sk[5] = 1;
    meq[6] = R(-2.0 / 3.0) * rho * uy;       Fb[6] = R(-2.0 / 3.0) * Fy; sk[6] = L.s_q;
    meq[7] = rho * uz;                       Fb[7] = Fz;                 sk[7] = 1;
    meq[8] = R(-2.0 / 3.0) * rho * uz;       Fb[8] = R(-2.0 / 3.0) * Fz; sk[8] = L.s_q;
    const R pxx = R(3) * ux * ux - uu, axx = R(2) * ux * Fx - uy * Fy - uz * Fz;
    const R pww = uy * uy - uz * uz, aww = uy * Fy - uz * Fz;
    meq[9] = rho * pxx;                      Fb[9] = R(2) * axx;         sk[9] = L.s_p;
    meq[10] = R(-0.5) * rho * pxx;           Fb[10] = -axx;              sk[10] = L.s_q;
    meq[11] = rho * pww;                     Fb[11] = R(2) * aww;        sk[11] = L.s_p;
    meq[12] = R(-0.5) * rho * pww;           Fb[12] = -aww;              sk[12] = L.s_q;
    meq[13] = rho * ux * uy;                 Fb[13] = ux * Fy + uy * Fx; sk[13] = L.s_p;
    meq[14] = rho * uy * uz;                 Fb[14] = uy * Fz + uz * Fy; sk[14] = L.s_p;
    meq[15] = rho * ux * uz;                 Fb[15] = ux * Fz + uz * Fx; sk[15] = L.s_p;
    meq[16] = 0;                             Fb[16] = 0;                 sk[16] = L.s_q;
    meq[17] = 0;                             Fb[17] = 0;                 sk[17] = L.s_q;
    meq[18] = 0;                             Fb[18] = 0;                 sk[18] = L.s_q;
    R dm[19];
#pragma unroll
    for (int kk = 0; kk < 19; ++kk)
        dm[kk] = (-sk[kk] * (m[kk] - meq[kk]) + (R(1) - R(0.5) * sk[kk]) * Fb[kk]) * R(1.0 / mnorm(kk));
    add_inverse19(dm, f);
}

// 12 sum_i varpi(|c_i|^2) psi(x + c_i) c_i (Eq. 9; varpi 1/6 on the axes, 1/12 on
// the diagonals) from pn(dx, dy, dz)
template <class R, class Get>
__device__ __forceinline__ void stencil3(Get pn, R* s) {
    const R axy = pn(1, 1, 0) - pn(-1, -1, 0), bxy = pn(1, -1, 0) - pn(-1, 1, 0);
    const R axz = pn(1, 0, 1) - pn(-1, 0, -1), bxz = pn(1, 0, -1) - pn(-1, 0, 1);
    const R ayz = pn(0, 1, 1) - pn(0, -1, -1), byz = pn(0, 1, -1) - pn(0, -1, 1);
    s[0] = R(2) * (pn(1, 0, 0) - pn(-1, 0, 0)) + ((axy + bxy) + (axz + bxz));
    s[1] = R(2) * (pn(0, 1, 0) - pn(0, -1, 0)) + ((axy - bxy) + (ayz + byz));
    s[2] = R(2) * (pn(0, 0, 1) - pn(0, 0, -1)) + ((axz - bxz) + (ayz - byz));
}

// Thermal stage: P^n (Eq. 20, with E = T dp/dT / (12 rho c_v) and c_s^2 grad T =
// -varsigma_1 times the first moments) and the D3Q7 MRT collision of the
// (deviation) populations g with source Q + S = rho c_v (P^n + (P^n - P^{n-1})/2)
template <bool UNIT, class R>
__device__ __forceinline__ R thermal7(const Lat3<R>& L, const R* g, R C, R E, R ux, R uy, R uz,
                                      R div12, R Pp, bool first, R* gs) {
    const R m1 = g[1] - g[2], m2 = g[3] - g[4], m3 = g[5] - g[6];
    const R s1 = g[1] + g[2], s2 = g[3] + g[4], s3 = g[5] + g[6];
    const R Td = g[0] + ((s1 + s2) + s3);
    const R Pn = L.vs1_cs2h * (ux * m1 + uy * m2 + uz * m3) - E * div12;
    const R dP = first ? Pn : Pn + R(0.5) * (Pn - Pp);
    if (UNIT) {
        // varsigma_3 = varsigma_4 = 1: only T and the first moments remain
        const R TQ = Td + C * dP;
        const R a = L.w7_1 * TQ;
        gs[0] = TQ - R(6) * a;      // what the others leave of T
        gs[1] = a + L.h_m * m1;
        gs[2] = a - L.h_m * m1;
        gs[3] = a + L.h_m * m2;
        gs[4] = a - L.h_m * m2;
        gs[5] = a + L.h_m * m3;
        gs[6] = a - L.h_m * m3;
    } else {
        // closed-form inverse of the moment matrix (rows 1, c_x, c_y, c_z,
        // |c|^2, c_x^2 - c_y^2, c_y^2 - c_z^2)
        const R Qs = C * dP;
        const R m4 = (s1 + s2) + s3, m5 = s1 - s2, m6 = s2 - s3;
        const R wd = L.w7_1 * R(6);
        const R t4 = m4 - L.vs3 * (m4 - wd * Td) + wd * Qs;
        const R t5 = m5 - L.vs4 * m5, t6 = m6 - L.vs4 * m6;
        const R b = (t4 - t5 + t6) * R(1.0 / 3.0);
        const R a = b + t5, c = b - t6;
        gs[0] = (Td + Qs) - t4;
        gs[1] = R(0.5) * a + L.h_m * m1;
        gs[2] = R(0.5) * a - L.h_m * m1;
        gs[3] = R(0.5) * b + L.h_m * m2;
        gs[4] = R(0.5) * b - L.h_m * m2;
        gs[5] = R(0.5) * c + L.h_m * m3;
        gs[6] = R(0.5) * c - L.h_m * m3;
    }
    return Pn;
}

__device__ __forceinline__ int wrapn(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
// any distance from the domain (tiles wider than a small domain wrap several times)
__device__ __forceinline__ int wrapm(int i, int n) { const int r = i % n; return r < 0 ? r + n : r; }

template <class R>
__device__ __forceinline__ size_t nid(const Dom3& D, int x, int y, int z) {
    return ((size_t)z * D.ny + y) * D.pitch + x;
}

// Element offsets from a node to its six axis neighbours, wrapped across the
// periodic seams; a lattice direction's offset is the sum of its components'.
// zlo / zhi: the node is next to the bottom / top wall.
struct Nbr {
    long long xp, xm, yp, ym, zp, zm;
    bool zlo, zhi;
};

__device__ __forceinline__ Nbr nbr_offsets(const Dom3& D, int x, int y, int z) {
    Nbr d;
    const long long P = D.pitch, S = (long long)D.ny * D.pitch;
    d.xp = x == D.nx - 1 ? -(long long)(D.nx - 1) : 1;
    d.xm = x == 0 ? (long long)(D.nx - 1) : -1;
    d.yp = y == D.ny - 1 ? -(long long)(D.ny - 1) * P : P;
    d.ym = y == 0 ? (long long)(D.ny - 1) * P : -P;
    d.zp = z == D.nz - 1 ? -(long long)(D.nz - 1) * S : S;
    d.zm = z == 0 ? (long long)(D.nz - 1) * S : -S;
    d.zlo = D.walls && z == 0;
    d.zhi = D.walls && z == D.nz - 1;
    return d;
}

// offset of the node at c = (cx, cy, cz) away (each component -1, 0 or 1)
__device__ __forceinline__ long long nbr_off(const Nbr& d, int cx, int cy, int cz) {
    long long o = 0;
    if (cx > 0) o += d.xp;
    if (cx < 0) o += d.xm;
    if (cy > 0) o += d.yp;
    if (cy < 0) o += d.ym;
    if (cz > 0) o += d.zp;
    if (cz < 0) o += d.zm;
    return o;
}

// the node c away lies beyond a wall
__device__ __forceinline__ bool nbr_solid(const Nbr& d, int cz) {
    return (cz < 0 && d.zlo) || (cz > 0 && d.zhi);
}

// ---------------------------------------------------------------------------
// psi of a node beyond a wall: the ghost layer, from rho / T of layers 1 and 2
template <class R>
__device__ R psi_ghost(const Dom3& D, const Phys<R>& P, int x, int y, int z, int* err) {
    const R* A = (const R*)D.aux;
    x = wrapn(x, D.nx);
    y = wrapn(y, D.ny);
    const int e = z < 0 ? 0 : 1;
    const int z1 = e == 0 ? 0 : D.nz - 1, z2 = e == 0 ? 1 : D.nz - 2;
    const R* rho = A + Q_RHO * D.plane;
    const R dx = rho[nid<R>(D, wrapn(x + 1, D.nx), y, z1)] - rho[nid<R>(D, wrapn(x - 1, D.nx), y, z1)];
    const R dy = rho[nid<R>(D, x, wrapn(y + 1, D.ny), z1)] - rho[nid<R>(D, x, wrapn(y - 1, D.ny), z1)];
    const R rg = (rho[nid<R>(D, x, y, z2)] + (R)D.rho_ref) + (R)D.cot * rsq(dx * dx + dy * dy);
    const R tg = A[Q_T * D.plane + nid<R>(D, x, y, z1)];   // the fluid node's temperature
    R q2, E;
    eos_node(P, rg, tg, &q2, &E);
    if (!(q2 >= R(0))) *err |= (q2 != q2) ? ERR_NONFINITE : ERR_PSI;
    return f_sqrt(q2);
}

// F_m from the psi of the 18 neighbours and F = F_m + F_b at node n
// (Eqs. 9, 11); S = 144 |F_m|^2 / (G psi)^2 for the sigma term
template <class R>
__device__ __forceinline__ void force_at(const Dom3& D, const Phys<R>& P, const Lat3<R>& L,
                                         int x, int y, int z, size_t n, const Nbr& nb,
                                         long long step, int* err, R* F, R* S) {
    const R* A = (const R*)D.aux;
    const R* psi_p = A + Q_PSI * D.plane;
    R s[3];
    // beyond a wall the neighbour is the ghost layer (Section 3.3)
    stencil3<R>([&](int cx, int cy, int cz) {
        return nbr_solid(nb, cz) ? psi_ghost<R>(D, P, x + cx, y + cy, z + cz, err)
                                 : psi_p[(size_t)((long long)n + nbr_off(nb, cx, cy, cz))];
    }, s);
    const R gp = P.negG_12 * psi_p[n];
    F[0] = gp * s[0];
    F[1] = gp * s[1];
    F[2] = gp * s[2];
    if (L.gravity != R(0)) {
        const R rho_ave = (R)(__ldcg(&D.ctl->mass[(step + 2) % 3]) * D.inv_n);
        F[2] -= L.gravity * ((A[Q_RHO * D.plane + n] + L.rho_ref) - rho_ave);
    }
    *S = s[0] * s[0] + s[1] * s[1] + s[2] * s[2];
}

// u of the read-out
template <class R>
__global__ void __launch_bounds__(128) k3_force(Dom3 D, Phys<R> P, Lat3<R> L) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= D.nx || y >= D.ny) return;
    R* A = (R*)D.aux;
    const size_t n = nid<R>(D, x, y, z);
    const Nbr nb = nbr_offsets(D, x, y, z);
    int err = 0;
    R F[3], S;
    force_at<R>(D, P, L, x, y, z, n, nb, __ldcg(&D.ctl->step), &err, F, &S);
    R u[3] = {0, 0, 0};
    if (!L.frozen_flow) {
        const R ir = f_rcp(A[Q_RHO * D.plane + n] + L.rho_ref);
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] = (A[(Q_JX + a) * D.plane + n] + R(0.5) * F[a]) * ir;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) A[(Q_UX + a) * D.plane + n] = u[a];
    if (err) atomicOr(&D.ctl->err, err);
}

// ---------------------------------------------------------------------------
// Step over nodes (the default in FP64), after k3_macro: k3_flow has the force,
// u and the flow collision, k3_thermal what needs the neighbours' u and 1/(rho
// c_v).  In FP64 both are bound by the FP64 pipe (84 % busy).  At unit rates
// the collision takes rho, j and the stresses k3_macro has formed, so that
// neither the moments are formed again from f (a collision kernel that did both
// lattices after a kernel for the force spent 49 of 353 FP64 operations per
// node on that) nor F passes through memory: 96^3 FP64 605 -> 540 us per step
// (FP32 on the same path, 128^3: 189 -> 163).
template <class R, bool UNIT>
__global__ void __launch_bounds__(128) k3_flow(Dom3 D, Phys<R> P, Lat3<R> L) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= D.nx || y >= D.ny) return;
    const long long step = __ldcg(&D.ctl->step);
    const int par = (int)(step & 1);
    R* A = (R*)D.aux;
    const size_t n = nid<R>(D, x, y, z);
    const Nbr nb = nbr_offsets(D, x, y, z);
    int err = 0;
    Mom3<R> m;
    m.rhod = A[Q_RHO * D.plane + n];
#pragma unroll
    for (int a = 0; a < 3; ++a) m.j[a] = A[(Q_JX + a) * D.plane + n];
    R F[3], S;
    force_at<R>(D, P, L, x, y, z, n, nb, step, &err, F, &S);
    const R rho = m.rhod + L.rho_ref, ir = f_rcp(rho);
    R u[3] = {0, 0, 0};
    if (!L.frozen_flow) {
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] = (m.j[a] + R(0.5) * F[a]) * ir;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) A[(Q_UX + a) * D.plane + n] = u[a];
    A[Q_IC * D.plane + n] = ir * P.inv_cv;
    if (err) atomicOr(&D.ctl->err, err);

    // ---- D3Q19 MRT collision, pushed to x + c_i (bounce-back through walls)
    const R* fc = (const R*)D.f[par] + fofs(n);
    R* fn = (R*)D.f[par ^ 1];
    R f[19];
    if (!UNIT || L.frozen_flow) {
#pragma unroll
        for (int i = 0; i < 19; ++i) f[i] = fc[i * XB];
    }
    if (L.frozen_flow) {
#pragma unroll
        for (int i = 0; i < 19; ++i) fn[fofs(n) + i * XB] = f[i];
        return;
    }
    if constexpr (UNIT) {
#pragma unroll
        for (int a = 0; a < 5; ++a) m.st[a] = A[(Q_S + a) * D.plane + n];
        collide19_unit(L, m, u, F, S, f);
    } else {
        collide19(L, rho, u, F, P.negG_12 * P.negG_12 * S, f);
    }
    static_for<19>([&](auto icn) {
        constexpr int i = decltype(icn)::value;
        if (nbr_solid(nb, qz(i)))
            fn[fofs(n) + qopp(i) * XB] = f[i];
        else
            fn[fofs((size_t)((long long)n + nbr_off(nb, qx(i), qy(i), qz(i)))) + i * XB] = f[i];
    });
}

template <class R, bool UNIT>
__global__ void __launch_bounds__(128) k3_thermal(Dom3 D, Phys<R> P, Lat3<R> L) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= D.nx || y >= D.ny) return;
    const long long step = __ldcg(&D.ctl->step);
    const int par = (int)(step & 1);
    const size_t n = nid<R>(D, x, y, z);
    const R* gc = (const R*)D.g[par];
    R* gn = (R*)D.g[par ^ 1];
    const R* A = (const R*)D.aux;
    const R rho = A[Q_RHO * D.plane + n] + L.rho_ref;
    const R u[3] = {A[Q_UX * D.plane + n], A[Q_UY * D.plane + n], A[Q_UZ * D.plane + n]};
    const size_t gno = gofs(n);
    R g[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) g[i] = gc[gno + i * XB];
    const Nbr nb = nbr_offsets(D, x, y, z);
    // 12 div u = 12 (1/c_s^2) sum_i w_i c_i . u(x + c_i); walls carry u = 0
    R dva = 0, dvd = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        if (nbr_solid(nb, qz(i))) continue;
        const size_t m = (size_t)((long long)n + nbr_off(nb, qx(i), qy(i), qz(i)));
        R& acc = qc2(i) == 1 ? dva : dvd;
        if (qx(i)) acc += R(qx(i)) * A[Q_UX * D.plane + m];
        if (qy(i)) acc += R(qy(i)) * A[Q_UY * D.plane + m];
        if (qz(i)) acc += R(qz(i)) * A[Q_UZ * D.plane + m];
    }
    const R C = rho * P.cv;
    R gs[7];
    const R Pn = thermal7<UNIT>(L, g, C, A[Q_E * D.plane + n], u[0], u[1], u[2], R(2) * dva + dvd,
                                ((const R*)D.P[par])[n], step == 0, gs);
    ((R*)D.P[par ^ 1])[n] = Pn;

    // weighted streaming (Eq. 39) from this node's side: g*_i lands on
    // x = y + c_i as g_i(x) + (g*_i - g_i(x)) / (rho(x) c_v), with g_i(x)
    // and rho(x) those of the current state; through a wall g*_i
    // returns to this node as the opposite direction, A = 2 w^ T_w - g*_i
    // (Dirichlet) or g*_i (adiabatic)
    if (L.frozen_thermal) {
#pragma unroll
        for (int i = 0; i < 7; ++i) gn[gno + i * XB] = g[i];
    } else {
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            if ((i == 5 && nb.zhi) || (i == 6 && nb.zlo)) {
                const int e = i == 5 ? 1 : 0, o = i == 5 ? 6 : 5;
                const R Ai = D.therm[e] == T_DIRICHLET ? L.tw2[e] - gs[i] : gs[i];
                gn[gno + o * XB] = g[o] + (Ai - g[o]) * A[Q_IC * D.plane + n];
            } else {
                const size_t m = (size_t)((long long)n + nbr_off(nb, hx(i), hy(i), hz(i)));
                const size_t gm = gofs(m) + i * XB;
                const R go = gc[gm];
                gn[gm] = go + (gs[i] - go) * A[Q_IC * D.plane + m];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// macroscopic fields of a node from its (deviation) populations
template <class R>
struct Fld3 {
    R rho, T, psi, E;
};
template <class R>
__device__ __forceinline__ void fields3(const Phys<R>& P, const Lat3<R>& L, R rhod, R Td, Fld3<R>& o,
                                        int* err) {
    o.rho = rhod + L.rho_ref;
    o.T = Td + L.T_ref;
    R q2;
    eos_node(P, o.rho, o.T, &q2, &o.E);
    if (!(q2 >= R(0))) *err |= (q2 != q2) ? ERR_NONFINITE : ERR_PSI;
    o.psi = f_sqrt(q2);
}
template <class R>
__device__ __forceinline__ R sum7(const R* g) {
    return g[0] + (((g[1] + g[2]) + (g[3] + g[4])) + (g[5] + g[6]));
}

// block sum of rho into the density ring (FP64), for the buoyancy of the
// next step
__device__ __forceinline__ void add_mass(const Dom3& D, double v, int slot) {
    __shared__ double red[4];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((t & 31) == 0) red[t >> 5] = v;
    __syncthreads();
    if (t == 0) massq_add(&D.ctl->massq[slot], red[0] + red[1] + red[2] + red[3], massq_scale(D.inv_n));
}

// Fields of the current state from its populations, into the planes, with
// its density sum into slot step % 3 for buoyancy.  want: W_STRESS the stress
// moments (which the collision at unit rates takes), W_T the
// temperature everywhere (else only next to the walls, for the ghost layer).
// Bound by its traffic, 26 populations read and 6 to 11 fields written.
enum { W_STRESS = 1, W_T = 2 };
template <class R>
__global__ void __launch_bounds__(128) k3_macro(Dom3 D, Phys<R> P, Lat3<R> L, int use_mass, int want) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    const bool in = x < D.nx && y < D.ny;
    double msum = 0.0;
    const long long step = __ldcg(&D.ctl->step);
    if (in) {
        const int par = (int)(step & 1);
        const size_t n = nid<R>(D, x, y, z);
        const R* fc = (const R*)D.f[par] + fofs(n);
        const R* gc = (const R*)D.g[par] + gofs(n);
        R f[19], g[7];
#pragma unroll
        for (int i = 0; i < 19; ++i) f[i] = __ldg(fc + i * XB);
#pragma unroll
        for (int i = 0; i < 7; ++i) g[i] = __ldg(gc + i * XB);
        int err = 0;
        Mom3<R> m;
        Fld3<R> o;
        moments3<true>(f, m);
        fields3(P, L, m.rhod, sum7(g), o, &err);
        R* A = (R*)D.aux + n;
        A[Q_RHO * D.plane] = m.rhod;
        A[Q_PSI * D.plane] = o.psi;
        A[Q_E * D.plane] = o.E;
#pragma unroll
        for (int a = 0; a < 3; ++a) A[(Q_JX + a) * D.plane] = m.j[a];
        if (want & W_STRESS) {
#pragma unroll
            for (int a = 0; a < 5; ++a) A[(Q_S + a) * D.plane] = m.st[a];
        }
        if ((want & W_T) || (D.walls && (z == 0 || z == D.nz - 1))) A[Q_T * D.plane] = o.T;
        if (err) atomicOr(&D.ctl->err, err);
        if (use_mass) msum = (double)o.rho;
    }
    if (use_mass) add_mass(D, in ? msum : 0.0, (int)(step % 3));
}

// end of a step: publish its density sum, clear the slot the next step
// accumulates into and advance the counter
__device__ __forceinline__ void end_step(Ctl* ctl, long long s, double qscale) {
    ctl->mass[s % 3] = massq_value(__ldcg(&ctl->massq[s % 3]), qscale);
    ctl->massq[(s + 1) % 3] = 0;
    ctl->step = s + 1;
}
__global__ void k3_advance(Ctl* ctl, double qscale) { end_step(ctl, ctl->step, qscale); }

// ---------------------------------------------------------------------------
// Marching step: after k3_macro has written the state's fields, one kernel does
// the rest of the step.  A CTA takes an xy tile of 32 x 8 nodes and a segment
// [z0, z1) of planes and marches k through the planes, the stages skewed so
// that each reads only planes its predecessors have finished (two barriers per
// plane):
//   psi(k) into shared memory on the tile + 2 (beyond a wall: the ghost-layer
//          psi, Section 3.3)
//   C(k-3) on the tile: div u, grad T, Q, P^n, S and the D3Q7 collision
//          (Eqs. 20, 24, 49-50); g*_i blended into the destination's
//          g(t+1) = g + (g* - g)/(rho c_v) (Eq. 39; anti-bounce-back at walls)
//   B(k-1) F_m, F, u and 1/(rho c_v) on the tile + 1 (Eqs. 9, 11); on the tile
//          the D3Q19 collision (Eq. 5) with f*_i pushed to x + c_i
//          (bounce-back at walls)
// Each node is collided by the CTA that owns it, which writes its
// post-collision populations straight to their destinations in f(t+1) and
// g(t+1).  At unit rates f itself is not read again: rho, j and the stresses
// are enough.  What the next iteration reads from memory is loaded into registers at the
// start of phase 2, so that it arrives while stage B computes.
//
// Bound by memory latency more than by bandwidth: it moves about 190 B per
// node (FP32), k3_macro 148.  256^3 FP32 per step: one kernel that recomputed
// the fields around each 16 x 16 tile from f 1390 us (its halo columns cost one
// sector per lane, L1 77 % busy), with the unit-rate collision and blocked
// populations 1316; this form with its loads at the end of phase 2 1206, psi
// and stage C's at the start 1123, stage B's too (two register sets) 988
// (17.0 GLUPS; k3_macro 346 us of it, at 7 TB/s).  Three CTAs per SM spill
// (80 registers) and take 1165.  32 x 8 tiles rather than 16 x 16: full 128-byte
// rows, and stencil reads without bank conflicts.
template <class R>
struct Tile3 {
    static constexpr int TX = 32, TY = 8, NT = 256;
    static constexpr int W2 = TX + 4, N2 = W2 * (TY + 4);   // tile + 2: psi
    static constexpr int W1 = TX + 2, N1 = W1 * (TY + 2);   // tile + 1: u, 1/(rho c_v)
    static constexpr int NB = N1 - TX * TY;                  // the ring around the tile
    static constexpr int ELEMS = 3 * N2 + 12 * N1;           // psi 3 planes, u 3 x 3, 1/(rho c_v) 3
    static constexpr size_t BYTES = (size_t)ELEMS * sizeof(R);
    static constexpr int MIN_BLOCKS = sizeof(R) == 4 ? 2 : 1;   // CTAs per SM
    static_assert(TX * TY == NT && N2 <= 2 * NT && NB <= NT, "one tile node per thread, psi in two passes");
};

template <class R, bool UNIT>
__global__ void __launch_bounds__(Tile3<R>::NT, Tile3<R>::MIN_BLOCKS)
k3_march(const __grid_constant__ Dom3 D, const __grid_constant__ Phys<R> P, const __grid_constant__ Lat3<R> L,
         int zseg) {
    using G = Tile3<R>;
    constexpr int TX = G::TX, TY = G::TY, NT = G::NT, W2 = G::W2, N2 = G::N2, W1 = G::W1, N1 = G::N1,
                  NB = G::NB;
    extern __shared__ __align__(16) unsigned char k3_smem[];
    R* const s_psi = reinterpret_cast<R*>(k3_smem);   // [3][N2]
    R* const s_u = s_psi + 3 * N2;                     // [3][3][N1]
    R* const s_ic = s_u + 9 * N1;                      // [3][N1] 1 / (rho c_v)

    const int tid = threadIdx.x;
    const int ntx = (D.nx + TX - 1) / TX;
    const int x0 = (int)(blockIdx.x % ntx) * TX, y0 = (int)(blockIdx.x / ntx) * TY;
    const int z0 = (int)blockIdx.y * zseg, z1 = min(D.nz, z0 + zseg);
    const long long step = __ldcg(&D.ctl->step);
    const int par = (int)(step & 1);
    const bool first = step == 0;
    const R* __restrict__ const fc = (const R*)D.f[par];
    R* __restrict__ const fnx = (R*)D.f[par ^ 1];
    const R* __restrict__ const gc = (const R*)D.g[par];
    R* __restrict__ const gnx = (R*)D.g[par ^ 1];
    const R* __restrict__ const Pc = (const R*)D.P[par];
    R* __restrict__ const Pnx = (R*)D.P[par ^ 1];
    const R* __restrict__ const A = (const R*)D.aux;
    const size_t ZS = (size_t)D.ny * D.pitch, PL = D.plane;
    const R rho_ave = L.gravity != R(0) ? (R)(__ldcg(&D.ctl->mass[(step + 2) % 3]) * D.inv_n) : R(0);

    // in-plane element offsets (32 bits: the host keeps larger planes on the
    // step over nodes), each the sum of a column and a row part
    auto fX = [&](int x) { return (unsigned)(x / XB) * (19u * XB) + (unsigned)(x % XB); };
    auto gX = [&](int x) { return (unsigned)(x / XB) * (7u * XB) + (unsigned)(x % XB); };
    const unsigned fP = 19u * (unsigned)D.pitch, gP = 7u * (unsigned)D.pitch;
    // the tile node this thread takes, its wrapped neighbour columns and rows
    // (a tile that reaches beyond the domain wraps onto it, as its halo does)
    const int cx = tid % TX, cy = tid / TX;
    const int gx = wrapm(x0 + cx, D.nx), gy = wrapm(y0 + cy, D.ny);
    const bool own = x0 + cx < D.nx && y0 + cy < D.ny;
    const int xm = gx == 0 ? D.nx - 1 : gx - 1, xp = gx == D.nx - 1 ? 0 : gx + 1;
    const int ym = gy == 0 ? D.ny - 1 : gy - 1, yp = gy == D.ny - 1 ? 0 : gy + 1;
    const unsigned fx0 = fX(gx), fxm = fX(xm), fxp = fX(xp);
    const unsigned fy0 = gy * fP, fym = ym * fP, fyp = yp * fP;
    const unsigned gx0 = gX(gx), gxm = gX(xm), gxp = gX(xp);
    const unsigned gy0 = gy * gP, gym = ym * gP, gyp = yp * gP;
    const unsigned oN = (unsigned)gy * D.pitch + gx;
    const int c2 = (cy + 2) * W2 + cx + 2, c1 = (cy + 1) * W1 + cx + 1;
    // its node of the ring around the tile (tid < NB) and its nodes of tile + 2
    int rx = 0, ry = 0;
    if (tid < W1) { rx = tid - 1; ry = -1; }
    else if (tid < 2 * W1) { rx = tid - W1 - 1; ry = TY; }
    else if (tid < 2 * W1 + TY) { rx = -1; ry = tid - 2 * W1; }
    else if (tid < NB) { rx = TX; ry = tid - 2 * W1 - TY; }
    const int r2 = (ry + 2) * W2 + rx + 2, r1 = (ry + 1) * W1 + rx + 1;
    const unsigned rN = (unsigned)wrapm(y0 + ry, D.ny) * D.pitch + wrapm(x0 + rx, D.nx);
    unsigned pN[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int a = tid + r * NT;
        pN[r] = a < N2 ? (unsigned)wrapm(y0 + a / W2 - 2, D.ny) * D.pitch + wrapm(x0 + a % W2 - 2, D.nx) : 0u;
    }

    int err = 0;
    // psi of the ghost layer beyond a wall at in-plane node n (Section 3.3): rho_ghost =
    // rho(layer 2) + tan(pi/2 - theta) |tangential difference of rho at layer 1|,
    // at the temperature of layer 1
    auto ghost = [&](unsigned n, bool lo) -> R {
        const int x = (int)(n % (unsigned)D.pitch), y = (int)(n / (unsigned)D.pitch);
        const size_t za = lo ? 0 : (size_t)(D.nz - 1) * ZS, zb = lo ? ZS : (size_t)(D.nz - 2) * ZS;
        const R* const rho = A + Q_RHO * PL;
        const size_t row = za + n - x;
        const R dx = rho[row + (x == D.nx - 1 ? 0 : x + 1)] - rho[row + (x == 0 ? D.nx - 1 : x - 1)];
        const R dy = rho[za + (size_t)(y == D.ny - 1 ? 0 : y + 1) * D.pitch + x] -
                     rho[za + (size_t)(y == 0 ? D.ny - 1 : y - 1) * D.pitch + x];
        R q2, E;
        eos_node(P, (rho[zb + n] + L.rho_ref) + (R)D.cot * rsq(dx * dx + dy * dy), A[Q_T * PL + za + n], &q2, &E);
        if (!(q2 >= R(0))) err |= (q2 != q2) ? ERR_NONFINITE : ERR_PSI;
        return f_sqrt(q2);
    };

    // ---- loads ahead: psi of plane k, what B needs of plane p, C of plane q
    R a_psi[2], b_o[9], b_r[4], c_g[7], c_t[6], c_P, c_rho, c_E;
    auto beyond = [&](int z) { return D.walls && (z < 0 || z >= D.nz); };
    auto load_psi = [&](int k, size_t zk) {
        if (k > z1 + 1) return;
        if (!beyond(k)) {
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (r == 0 || tid + NT < N2) a_psi[r] = __ldg(A + Q_PSI * PL + zk + pN[r]);
        } else if (k == -1 || k == D.nz) {
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (r == 0 || tid + NT < N2) a_psi[r] = ghost(pN[r], k < 0);
        }
    };
    auto b_active = [&](int p) { return p >= z0 - 1 && p <= z1 && !beyond(p); };
    auto load_b = [&](int p, size_t zp, R* b_o, R* b_r) {
        if (!b_active(p)) return;
        const R* const a = A + zp + oN;
        b_o[0] = __ldg(a + Q_RHO * PL);
#pragma unroll
        for (int i = 0; i < 3; ++i) b_o[1 + i] = __ldg(a + (Q_JX + i) * PL);
        if (UNIT && p >= z0 && p < z1) {
#pragma unroll
            for (int i = 0; i < 5; ++i) b_o[4 + i] = __ldg(a + (Q_S + i) * PL);
        }
        if (tid < NB) {
            const R* const b = A + zp + rN;
            b_r[0] = __ldg(b + Q_RHO * PL);
#pragma unroll
            for (int i = 0; i < 3; ++i) b_r[1 + i] = __ldg(b + (Q_JX + i) * PL);
        }
    };
    auto load_c = [&](int q) {
        if (!(q >= z0 && q < z1 && own)) return;
        const size_t zq = (size_t)q * ZS;
        const size_t zp = q == D.nz - 1 ? 0 : zq + ZS, zm = q == 0 ? (size_t)(D.nz - 1) * ZS : zq - ZS;
        const R* const g = gc + zq * 7;
#pragma unroll
        for (int i = 0; i < 7; ++i) c_g[i] = __ldg(g + (gy0 + gx0) + i * XB);
        // g_i of the nodes the blend goes to
        c_t[0] = __ldg(g + (gy0 + gxp) + 1 * XB);
        c_t[1] = __ldg(g + (gy0 + gxm) + 2 * XB);
        c_t[2] = __ldg(g + (gyp + gx0) + 3 * XB);
        c_t[3] = __ldg(g + (gym + gx0) + 4 * XB);
        c_t[4] = __ldg(gc + zp * 7 + (gy0 + gx0) + 5 * XB);
        c_t[5] = __ldg(gc + zm * 7 + (gy0 + gx0) + 6 * XB);
        c_P = __ldg(Pc + zq + oN);
        c_rho = __ldg(A + Q_RHO * PL + zq + oN);
        c_E = __ldg(A + Q_E * PL + zq + oN);
    };

    int zk = wrapm(z0 - 2, D.nz);    // plane k, wrapped
    int k3 = 0;                      // ring slot of plane k
    load_psi(z0 - 2, (size_t)zk * ZS);
    for (int k = z0 - 2; k <= z1 + 2; ++k) {
        const int km = k3 == 0 ? 2 : k3 - 1, kp = k3 == 2 ? 0 : k3 + 1;   // slots of k - 1, k - 2 (= k + 1)
        // ================= phase 1: psi(k), C(k - 3)
        if (k <= z1 + 1) {
            R* const ps = s_psi + k3 * N2 + tid;
            ps[0] = a_psi[0];
            if (tid + NT < N2) ps[NT] = a_psi[1];
        }
        {
            const int q = k - 3;
            if (q >= z0 && q < z1 && own) {
                const size_t zq = (size_t)q * ZS;
                const bool lo_wall = D.walls && q == 0, hi_wall = D.walls && q == D.nz - 1;
                const size_t zp = q == D.nz - 1 ? 0 : zq + ZS, zm = q == 0 ? (size_t)(D.nz - 1) * ZS : zq - ZS;
                // planes q - 1, q, q + 1 = k - 4, k - 3, k - 2
                const R* const um = s_u + km * 3 * N1 + c1;
                const R* const u0 = s_u + k3 * 3 * N1 + c1;
                const R* const up = s_u + kp * 3 * N1 + c1;
                // 12 div u = 12 (1/c_s^2) sum_i w_i c_i . u(x + c_i); walls carry u = 0
                R dva = 0, dvd = 0;
                auto div_plane = [&](const R* u, int dz) {
#pragma unroll
                    for (int i = 1; i < 19; ++i) {
                        if (qz(i) != dz) continue;
                        const R* us = u + qy(i) * W1 + qx(i);
                        R& acc = qc2(i) == 1 ? dva : dvd;
                        if (qx(i)) acc += R(qx(i)) * us[0];
                        if (qy(i)) acc += R(qy(i)) * us[N1];
                        if (qz(i)) acc += R(qz(i)) * us[2 * N1];
                    }
                };
                div_plane(u0, 0);
                if (!lo_wall) div_plane(um, -1);
                if (!hi_wall) div_plane(up, 1);
                R gs[7];
                Pnx[zq + oN] = thermal7<UNIT>(L, c_g, (c_rho + L.rho_ref) * P.cv, c_E, u0[0], u0[N1], u0[2 * N1],
                                              R(2) * dva + dvd, c_P, first, gs);
                // weighted streaming (Eq. 39) from this node's side: g*_i lands on
                // x = y + c_i as g_i(x) + (g*_i - g_i(x)) / (rho(x) c_v) of the
                // current state; through a wall it returns here as the opposite
                // direction, A = 2 w^ T_w - g*_i (Dirichlet) or g*_i (adiabatic)
                R* const go = gnx + zq * 7;
                const unsigned o = gy0 + gx0;
                if (L.frozen_thermal) {
#pragma unroll
                    for (int i = 0; i < 7; ++i) go[o + i * XB] = c_g[i];
                } else {
                    const R* const i0 = s_ic + k3 * N1 + c1;
                    const R ic = i0[0];
                    go[o] = c_g[0] + (gs[0] - c_g[0]) * ic;
                    go[(gy0 + gxp) + 1 * XB] = c_t[0] + (gs[1] - c_t[0]) * i0[1];
                    go[(gy0 + gxm) + 2 * XB] = c_t[1] + (gs[2] - c_t[1]) * i0[-1];
                    go[(gyp + gx0) + 3 * XB] = c_t[2] + (gs[3] - c_t[2]) * i0[W1];
                    go[(gym + gx0) + 4 * XB] = c_t[3] + (gs[4] - c_t[3]) * i0[-W1];
                    if (hi_wall) {
                        const R a = D.therm[1] == T_DIRICHLET ? L.tw2[1] - gs[5] : gs[5];
                        go[o + 6 * XB] = c_g[6] + (a - c_g[6]) * ic;
                    } else {
                        gnx[zp * 7 + o + 5 * XB] = c_t[4] + (gs[5] - c_t[4]) * s_ic[kp * N1 + c1];
                    }
                    if (lo_wall) {
                        const R a = D.therm[0] == T_DIRICHLET ? L.tw2[0] - gs[6] : gs[6];
                        go[o + 5 * XB] = c_g[5] + (a - c_g[5]) * ic;
                    } else {
                        gnx[zm * 7 + o + 6 * XB] = c_t[5] + (gs[6] - c_t[5]) * s_ic[km * N1 + c1];
                    }
                }
            }
        }
        __syncthreads();

        // ================= phase 2: B(k - 1)
        const size_t zb = (size_t)zk * ZS;
        zk = zk + 1 == D.nz ? 0 : zk + 1;
        load_psi(k + 1, (size_t)zk * ZS);
        load_c(k - 2);
        R n_o[9], n_r[4];
        load_b(k, zb, n_o, n_r);
        {
            const int p = k - 1;
            if (b_active(p)) {
                const R* const psm = s_psi + kp * N2;    // plane k - 2
                const R* const ps0 = s_psi + km * N2;
                const R* const psp = s_psi + k3 * N2;
                R* const uB = s_u + km * 3 * N1;
                R* const iB = s_ic + km * N1;
                // F and u of a node of tile + 1; returns |12 s|^2 of the stencil
                auto force = [&](int i2, int i1, R rho, const R* j, R* F, R* u) -> R {
                    R s[3];
                    stencil3<R>([&](int dx, int dy, int dz) {
                        return (dz < 0 ? psm : (dz > 0 ? psp : ps0))[i2 + dy * W2 + dx];
                    }, s);
                    const R gpsi = P.negG_12 * ps0[i2];
#pragma unroll
                    for (int a = 0; a < 3; ++a) F[a] = gpsi * s[a];
                    F[2] -= L.gravity * (rho - rho_ave);
                    const R ir = f_rcp(rho);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        u[a] = L.frozen_flow ? R(0) : (j[a] + R(0.5) * F[a]) * ir;
                        uB[a * N1 + i1] = u[a];
                    }
                    iB[i1] = ir * P.inv_cv;
                    return s[0] * s[0] + s[1] * s[1] + s[2] * s[2];
                };
                R F[3], u[3];
                if (tid < NB) force(r2, r1, b_r[0] + L.rho_ref, b_r + 1, F, u);
                const R rho = b_o[0] + L.rho_ref;
                const R S = force(c2, c1, rho, b_o + 1, F, u);
                // the tile node: collide it if this CTA owns it
                if (p >= z0 && p < z1 && own) {
                    const size_t zc = (size_t)p * ZS;
                    R* const b0 = fnx + zc * 19;
                    R f[19];
                    if (!UNIT || L.frozen_flow) {
                        const R* const fl = fc + zc * 19 + (fy0 + fx0);
#pragma unroll
                        for (int i = 0; i < 19; ++i) f[i] = fl[i * XB];
                    }
                    if (L.frozen_flow) {
#pragma unroll
                        for (int i = 0; i < 19; ++i) b0[(fy0 + fx0) + i * XB] = f[i];
                    } else {
                        if constexpr (UNIT) {
                            Mom3<R> m;
                            m.rhod = b_o[0];
#pragma unroll
                            for (int a = 0; a < 3; ++a) m.j[a] = b_o[1 + a];
#pragma unroll
                            for (int a = 0; a < 5; ++a) m.st[a] = b_o[4 + a];
                            collide19_unit(L, m, u, F, S, f);
                        } else {
                            collide19(L, rho, u, F, P.negG_12 * P.negG_12 * S, f);
                        }
                        // push to x + c_i; through a wall f*_i returns as f_opp(i)
                        const bool lo_wall = D.walls && p == 0, hi_wall = D.walls && p == D.nz - 1;
                        R* const bp = fnx + (p == D.nz - 1 ? 0 : zc + ZS) * 19;
                        R* const bm = fnx + (p == 0 ? (size_t)(D.nz - 1) * ZS : zc - ZS) * 19;
                        static_for<19>([&](auto icn) {
                            constexpr int i = decltype(icn)::value;
                            const unsigned o = (qx(i) > 0 ? fxp : (qx(i) < 0 ? fxm : fx0)) +
                                               (qy(i) > 0 ? fyp : (qy(i) < 0 ? fym : fy0));
                            if ((qz(i) < 0 && lo_wall) || (qz(i) > 0 && hi_wall))
                                b0[(fy0 + fx0) + qopp(i) * XB] = f[i];
                            else
                                (qz(i) > 0 ? bp : (qz(i) < 0 ? bm : b0))[o + i * XB] = f[i];
                        });
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) b_o[i] = n_o[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) b_r[i] = n_r[i];
        __syncthreads();
        k3 = kp;
    }

    if (err) atomicOr(&D.ctl->err, err);
    // the last CTA ends the step
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(&D.ctl->done, 1) == (int)(gridDim.x * gridDim.y) - 1) {
            __threadfence();
            end_step(D.ctl, step, massq_scale(D.inv_n));
            D.ctl->done = 0;
        }
    }
}

// populations f = f^eq(rho, u), g = w^ T as deviations; P = 0
template <class R>
__global__ void k3_init(Dom3 D, Lat3<R> L, const double* rho, const double* ux,
                        const double* uy, const double* uz, const double* T) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= D.nx || y >= D.ny) return;
    const size_t h = ((size_t)z * D.ny + y) * D.nx + x, n = nid<R>(D, x, y, z);
    R* f = (R*)D.f[0] + fofs(n);
    R* g = (R*)D.g[0] + gofs(n);
    const double r = rho[h], a = ux[h], b = uy[h], c = uz[h], t = T[h];
    const double uu = a * a + b * b + c * c;
#pragma unroll 19
    for (int i = 0; i < 19; ++i) {
        const double cu = qx(i) * a + qy(i) * b + qz(i) * c;
        const double fe = qw(i) * r * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
        f[i * XB] = (R)(fe - qw(i) * D.rho_ref);
    }
    const double w0 = (double)L.w7_0, w1 = (double)L.w7_1;
#pragma unroll 19
    for (int i = 0; i < 7; ++i) g[i * XB] = (R)((i == 0 ? w0 : w1) * (t - D.T_ref));
    ((R*)D.P[0])[n] = R(0);
}

// state -> host-layout doubles: fields (what 0: rho, u, T; 2: and |u|) or, what 1,
// absolute populations
template <class R>
__global__ void k3_export(Dom3 D, Lat3<R> L, int what, double* out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= D.nx || y >= D.ny) return;
    const size_t N = (size_t)D.nx * D.ny * D.nz;
    const size_t h = ((size_t)z * D.ny + y) * D.nx + x, n = nid<R>(D, x, y, z);
    const int par = (int)(__ldcg(&D.ctl->step) & 1);
    if (what != 1) {
        const R* A = (const R*)D.aux + n;
        const double ux = widen(A[Q_UX * D.plane]), uy = widen(A[Q_UY * D.plane]),
                     uz = widen(A[Q_UZ * D.plane]);
        out[0 * N + h] = widen(A[Q_RHO * D.plane]) + D.rho_ref;
        out[1 * N + h] = ux;
        out[2 * N + h] = uy;
        out[3 * N + h] = uz;
        out[4 * N + h] = widen(A[Q_T * D.plane]);
        if (what == 2) out[5 * N + h] = sqrt(ux * ux + uy * uy + uz * uz);   // for the diagnostics
    } else {
        const R* f = (const R*)D.f[par] + fofs(n);
        const R* g = (const R*)D.g[par] + gofs(n);
        for (int i = 0; i < 19; ++i) out[i * N + h] = (double)f[i * XB] + qw(i) * D.rho_ref;
        for (int i = 0; i < 7; ++i)
            out[(19 + i) * N + h] = (double)g[i * XB] +
                                    (double)(i == 0 ? L.w7_0 : L.w7_1) * D.T_ref;
        out[26 * N + h] = (double)((const R*)D.P[par])[n];
    }
}

}  // namespace
}  // namespace lbm

using namespace lbm;

struct lbm3d_ctx {
    int nx = 0, ny = 0, nz = 0, prec = 1;
    lbm_params params;
    lbm3d_bc bc;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    void* mem = nullptr;
    Ctl* ctl = nullptr;
    Dom3 D;
    cudaGraphExec_t graph = nullptr;
    bool fused = true;       // marching step (else the step over nodes)
    int zseg = 0;            // planes per CTA of the marching step
    long long step = 0;
    bool initialized = false;
    bool unseen = false;     // the step over nodes has made a state whose fields are not formed yet
    int sticky = LBM_OK;
    std::string err;
    double* host_buf = nullptr;   // device doubles: 27 N (export), reused
    void* diag_scratch = nullptr;
    double* diag_out = nullptr;
    double* zeros = nullptr;
};

namespace {

size_t pitch_for(int nx) { return ((size_t)nx + 31) / 32 * 32; }

size_t bytes_for(int nx, int ny, int nz, int prec) {
    const size_t es = prec == LBM_FP64 ? 8 : 4;
    const size_t plane = pitch_for(nx) * ny * nz;
    // f 2 x 19, g 2 x 7, P 2, the per-node planes 15, and two layers that no kernel
    // uses but the published size counts
    return plane * es * (38 + 14 + 2 + Q_N) + 2 * pitch_for(nx) * ny * es;
}

// planes per CTA of the marching step.  A segment costs about three planes
// beyond its own, so a domain whose tiles leave room takes the shortest segments
// that still fit the resident CTAs in one round (64^3 FP32: 4 planes 23.4 us per
// step, 2 planes 27.9, 8 planes 26.4; 128^3: 32 planes 136 us, 16 planes 144; 72
// x 50 x 61 between walls: 6 planes 37 us, 4 planes 44, 16 planes 47).  Larger
// domains take 32 planes (256^3: 988 us; 48 planes 998, 64 planes 1039).
int auto_zseg(int nx, int ny, int nz, int prec) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        sms = 148;
    const int tx = Tile3<float>::TX, ty = Tile3<float>::TY;
    const long long tiles = (long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
    const long long slots = (long long)sms * (prec == LBM_FP64 ? Tile3<double>::MIN_BLOCKS
                                                              : Tile3<float>::MIN_BLOCKS);
    const long long nseg = slots / tiles;
    const long long zs = nseg >= 1 ? (nz + nseg - 1) / nseg : nz;
    return (int)(zs <= 48 ? zs : 32);
}

int set_err3(lbm3d_ctx* c, int code, const char* msg) {
    if (c) c->err = msg;
    return code;
}

int cuda_err3(lbm3d_ctx* c, cudaError_t e, const char* where) {
    if (e == cudaSuccess) return LBM_OK;
    if (c) c->err = std::string(where) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
}

// one thread per node
dim3 blk3() { return dim3(32, 4, 1); }
dim3 grd3(const lbm3d_ctx* c) { return dim3((c->nx + 31) / 32, (c->ny + 3) / 4, c->nz); }

bool unit3(const lbm3d_ctx* c) { return unit_rates(phys_of(c->params)); }

// the marching kernel addresses a plane's populations with 32-bit element offsets;
// larger planes (more than 113 million nodes) take the step over nodes
bool march_fits(const lbm3d_ctx* c) {
    return (unsigned long long)c->ny * c->D.pitch * 19ull < (1ull << 31);
}

template <class R>
int launch_march(lbm3d_ctx* c) {
    using G = Tile3<R>;
    Phys<R> P = make_phys<R>(phys_of(c->params));
    Lat3<R> L = make_lat3<R>(c->params, c->D);
    const dim3 grid((unsigned)(((c->nx + G::TX - 1) / G::TX) * ((c->ny + G::TY - 1) / G::TY)),
                    (unsigned)((c->nz + c->zseg - 1) / c->zseg));
    const bool unit = unit3(c);
    k3_macro<R><<<grd3(c), blk3(), 0, c->stream>>>(c->D, P, L, c->params.gravity != 0.0, unit ? W_STRESS : 0);
    if (unit) k3_march<R, true><<<grid, G::NT, G::BYTES, c->stream>>>(c->D, P, L, c->zseg);
    else k3_march<R, false><<<grid, G::NT, G::BYTES, c->stream>>>(c->D, P, L, c->zseg);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// the fields of the current state that the read-out needs (rho, u, T)
template <class R>
void launch_fields(lbm3d_ctx* c, int what) {
    const Phys<R> P = make_phys<R>(phys_of(c->params));
    const Lat3<R> L = make_lat3<R>(c->params, c->D);
    k3_macro<R><<<grd3(c), blk3(), 0, c->stream>>>(c->D, P, L, 0, W_T);
    k3_force<R><<<grd3(c), blk3(), 0, c->stream>>>(c->D, P, L);
    k3_export<R><<<grd3(c), blk3(), 0, c->stream>>>(c->D, L, what, c->host_buf);
}

template <class R>
int launch_step(lbm3d_ctx* c) {
    if (c->fused && march_fits(c)) return launch_march<R>(c);
    Phys<R> P = make_phys<R>(phys_of(c->params));
    Lat3<R> L = make_lat3<R>(c->params, c->D);
    const dim3 b = blk3(), g = grd3(c);
    const bool unit = unit3(c);
    k3_macro<R><<<g, b, 0, c->stream>>>(c->D, P, L, c->params.gravity != 0.0, unit ? W_STRESS : 0);
    if (unit) {
        k3_flow<R, true><<<g, b, 0, c->stream>>>(c->D, P, L);
        k3_thermal<R, true><<<g, b, 0, c->stream>>>(c->D, P, L);
    } else {
        k3_flow<R, false><<<g, b, 0, c->stream>>>(c->D, P, L);
        k3_thermal<R, false><<<g, b, 0, c->stream>>>(c->D, P, L);
    }
    k3_advance<<<1, 1, 0, c->stream>>>(c->ctl, massq_scale(c->D.inv_n));
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int step_once(lbm3d_ctx* c) { return c->prec == LBM_FP64 ? launch_step<double>(c) : launch_step<float>(c); }

int check3(lbm3d_ctx* c) {
    Ctl h;
    cudaError_t e = cudaMemcpyAsync(&h, c->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_err3(c, e, "reading the control block");
    if (h.err && c->sticky == LBM_OK) {
        c->sticky = (h.err & ERR_PSI) ? LBM_EPSI : LBM_ENONFINITE;
        c->err = c->sticky == LBM_EPSI ? "psi^2 < 0 at some node" : "non-finite density or temperature";
    }
    return c->sticky;
}

// As check3, for the state the last step made.  The step over nodes forms and
// checks the fields of a state when it starts from it; here they are formed for
// the check alone.  (The marching step reports a state with the step after it.)
int check_state(lbm3d_ctx* c) {
    if (c->unseen && c->sticky == LBM_OK) {
        if (c->prec == LBM_FP64)
            k3_macro<double><<<grd3(c), blk3(), 0, c->stream>>>(c->D, make_phys<double>(phys_of(c->params)),
                                                                make_lat3<double>(c->params, c->D), 0, 0);
        else
            k3_macro<float><<<grd3(c), blk3(), 0, c->stream>>>(c->D, make_phys<float>(phys_of(c->params)),
                                                               make_lat3<float>(c->params, c->D), 0, 0);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_err3(c, e, "fields kernel");
        c->unseen = false;
    }
    return check3(c);
}

int ensure_buf(lbm3d_ctx* c) {
    if (c->host_buf) return LBM_OK;
    const size_t N = (size_t)c->nx * c->ny * c->nz;
    cudaError_t e = cudaMalloc(&c->host_buf, 27 * N * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&c->diag_scratch, diag_scratch_bytes((long long)N));
    if (e == cudaSuccess) e = cudaMemset(c->diag_scratch, 0, diag_scratch_bytes((long long)N));
    if (e == cudaSuccess) e = cudaMalloc(&c->diag_out, 16 * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&c->zeros, N * sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(c->zeros, 0, N * sizeof(double));
    return cuda_err3(c, e, "cudaMalloc(export buffers)");
}

// current fields (rho, u, T; what = 2: |u| too) into host_buf[0 .. 6N)
int export_fields(lbm3d_ctx* c, int what) {
    int rc = ensure_buf(c);
    if (rc) return rc;
    if (c->prec == LBM_FP64) launch_fields<double>(c, what);
    else launch_fields<float>(c, what);
    c->unseen = false;
    return cuda_err3(c, cudaGetLastError(), "field export");
}

}  // namespace

extern "C" {

size_t lbm3d_state_bytes(int nx, int ny, int nz, int prec) {
    if (nx < 1 || ny < 1 || nz < 1 || (prec != LBM_FP64 && prec != LBM_FP32)) return 0;
    return bytes_for(nx, ny, nz, prec);
}

int lbm3d_create(int nx, int ny, int nz, const lbm_params* params, const lbm3d_bc* bc, int prec,
                 void* stream, lbm3d_ctx** out) {
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (nx < 1 || ny < 1 || nz < 1 || !params || !bc || (prec != LBM_FP64 && prec != LBM_FP32))
        return LBM_EINVAL;
    if (nx > 65535 || ny > 65535 || nz > 65535) return LBM_EINVAL;
    if (bc->flow_z != LBM_PERIODIC && bc->flow_z != LBM_WALL) return LBM_EINVAL;
    for (int e = 0; e < 2; ++e) {
        if (bc->therm[e] < 0 || bc->therm[e] > 2) return LBM_EINVAL;
        if ((bc->flow_z == LBM_PERIODIC) != (bc->therm[e] == LBM_T_PERIODIC)) return LBM_EINVAL;
    }
    if (bc->flow_z == LBM_WALL && nz < 2) return LBM_EINVAL;
    if (!(params->cv > 0) || !(params->nu > 0) || !(params->lambda > 0) ||
        !(params->w_dot > 0 && params->w_dot < 1) || params->G == 0.0 || !(params->b > 0) ||
        !(params->s_e > 0 && params->s_e < 2))
        return LBM_EINVAL;
    lbm3d_ctx* c = new (std::nothrow) lbm3d_ctx();
    if (!c) return LBM_ENOMEM;
    c->nx = nx;
    c->ny = ny;
    c->nz = nz;
    c->prec = prec;
    c->params = *params;
    c->bc = *bc;
    cudaError_t e = cudaSuccess;
    if (stream) {
        c->stream = (cudaStream_t)stream;
    } else {
        e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
        c->own_stream = e == cudaSuccess;
    }
    const size_t total = bytes_for(nx, ny, nz, prec);
    if (e == cudaSuccess) e = cudaMalloc(&c->mem, total);
    if (e == cudaSuccess) e = cudaMalloc(&c->ctl, sizeof(Ctl));
    if (e == cudaSuccess) e = cudaMemset(c->ctl, 0, sizeof(Ctl));
    if (e != cudaSuccess) {
        const int rc = e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
        lbm3d_destroy(c);
        return rc;
    }
    const size_t es = prec == LBM_FP64 ? 8 : 4;
    const size_t plane = pitch_for(nx) * ny * nz;
    char* m = (char*)c->mem;
    Dom3& D = c->D;
    memset(&D, 0, sizeof(D));
    size_t off = 0;
    for (int p = 0; p < 2; ++p) { D.f[p] = m + off; off += 19 * plane * es; }
    for (int p = 0; p < 2; ++p) { D.g[p] = m + off; off += 7 * plane * es; }
    for (int p = 0; p < 2; ++p) { D.P[p] = m + off; off += plane * es; }
    D.aux = m + off;
    D.ctl = c->ctl;
    D.nx = nx;
    D.ny = ny;
    D.nz = nz;
    D.pitch = (int)pitch_for(nx);
    D.plane = plane;
    D.walls = bc->flow_z == LBM_WALL;
    D.therm[0] = bc->therm[0];
    D.therm[1] = bc->therm[1];
    D.T_edge[0] = bc->T_edge[0];
    D.T_edge[1] = bc->T_edge[1];
    D.cot = tan(M_PI / 2.0 - bc->theta_deg * M_PI / 180.0);
    D.rho_ref = 1.0;
    D.T_ref = 0.0;
    D.inv_n = 1.0 / ((double)nx * ny * nz);
    c->zseg = auto_zseg(nx, ny, nz, prec);
    // the marching step is the faster in FP32 (72 x 50 x 61 34.5 against 36.6 us,
    // 128^3 136 against 162, 256^3 983 against 1256); in FP64, bound by the FP64 pipe, its one CTA per SM
    // keeps that pipe less busy (96^3 583 against 514 us)
    c->fused = prec == LBM_FP32;
    auto smem = [&](auto kernel, size_t bytes) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    if (prec == LBM_FP64) {
        smem(k3_march<double, true>, Tile3<double>::BYTES);
        smem(k3_march<double, false>, Tile3<double>::BYTES);
    } else {
        smem(k3_march<float, true>, Tile3<float>::BYTES);
        smem(k3_march<float, false>, Tile3<float>::BYTES);
    }
    // the pitch padding is never read, but keep it defined
    if (e == cudaSuccess) e = cudaMemset(c->mem, 0, total);
    if (e != cudaSuccess) {
        lbm3d_destroy(c);
        return LBM_ECUDA;
    }
    *out = c;
    return LBM_OK;
}

int lbm3d_init_fields(lbm3d_ctx* c, const double* rho, const double* ux, const double* uy,
                      const double* uz, const double* T) {
    if (!c || !rho || !ux || !uy || !uz || !T) return LBM_EINVAL;
    const size_t N = (size_t)c->nx * c->ny * c->nz;
    int rc = ensure_buf(c);
    if (rc) return rc;
    const double* src[5] = {rho, ux, uy, uz, T};
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 5 && e == cudaSuccess; ++k)
        e = cudaMemcpyAsync(c->host_buf + k * N, src[k], N * sizeof(double), cudaMemcpyHostToDevice,
                            c->stream);
    // storage references from device sums (fixed summation order)
    double sums[2];
    if (e == cudaSuccess && sum2_launch(c->host_buf, c->host_buf + 4 * N, (long long)N,
                                        c->diag_out + 8, c->diag_scratch, c->stream))
        e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(sums, c->diag_out + 8, sizeof(sums), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_err3(c, e, "field sums");
    c->D.rho_ref = c->params.rho_ref > 0 ? c->params.rho_ref : sums[0] / (double)N;
    c->D.T_ref = c->params.T_ref > 0 ? c->params.T_ref : sums[1] / (double)N;
    Ctl h;
    memset(&h, 0, sizeof(h));
    if (e == cudaSuccess) e = cudaMemcpyAsync(c->ctl, &h, sizeof(h), cudaMemcpyHostToDevice, c->stream);
    if (e != cudaSuccess) return cuda_err3(c, e, "copying the initial fields");
    const dim3 b = blk3(), g = grd3(c);
    const int um = c->params.gravity != 0.0;
    if (c->prec == LBM_FP64) {
        k3_init<double><<<g, b, 0, c->stream>>>(c->D, make_lat3<double>(c->params, c->D), c->host_buf,
                                                c->host_buf + N, c->host_buf + 2 * N,
                                                c->host_buf + 3 * N, c->host_buf + 4 * N);
        k3_macro<double><<<g, b, 0, c->stream>>>(c->D, make_phys<double>(phys_of(c->params)),
                                                 make_lat3<double>(c->params, c->D), um, 0);
    } else {
        k3_init<float><<<g, b, 0, c->stream>>>(c->D, make_lat3<float>(c->params, c->D), c->host_buf,
                                               c->host_buf + N, c->host_buf + 2 * N,
                                               c->host_buf + 3 * N, c->host_buf + 4 * N);
        k3_macro<float><<<g, b, 0, c->stream>>>(c->D, make_phys<float>(phys_of(c->params)),
                                                make_lat3<float>(c->params, c->D), um, 0);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_err3(c, e, "init kernels");
    // the initial density sum (accumulated into massq[0], which step 0 adds to
    // again) is read by step 0 from slot 2 ((0 - 1) mod 3)
    e = cudaStreamSynchronize(c->stream);
    if (e == cudaSuccess && um) {
        long long q0 = 0;
        e = cudaMemcpy(&q0, &c->ctl->massq[0], sizeof(q0), cudaMemcpyDeviceToHost);
        const double m0 = massq_value(q0, massq_scale(c->D.inv_n));
        if (e == cudaSuccess) e = cudaMemset(&c->ctl->massq[0], 0, sizeof(q0));
        if (e == cudaSuccess) e = cudaMemcpy(&c->ctl->mass[2], &m0, sizeof(double), cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) return cuda_err3(c, e, "lbm3d_init_fields");
    if (c->graph) cudaGraphExecDestroy(c->graph);
    c->graph = nullptr;   // the launch arguments carry rho_ref / T_ref
    c->step = 0;
    c->unseen = false;
    c->sticky = LBM_OK;
    c->initialized = true;
    c->err.clear();
    return check3(c);
}

int lbm3d_step(lbm3d_ctx* c, int n) {
    if (!c || n < 0) return LBM_EINVAL;
    if (!c->initialized) return set_err3(c, LBM_ESTATE, "lbm3d_step before lbm3d_init_fields");
    if (c->sticky) return c->sticky;
    if (n == 0) return LBM_OK;
    c->unseen = !(c->fused && march_fits(c));
    const int kLen = 32;
    int left = n;
    if (left >= kLen) {
        if (!c->graph) {
            cudaGraph_t g;
            cudaError_t e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
            if (e != cudaSuccess) return cuda_err3(c, e, "cudaStreamBeginCapture");
            for (int i = 0; i < kLen; ++i) step_once(c);
            e = cudaStreamEndCapture(c->stream, &g);
            if (e != cudaSuccess) return cuda_err3(c, e, "cudaStreamEndCapture");
            e = cudaGraphInstantiate(&c->graph, g, 0);
            cudaGraphDestroy(g);
            if (e != cudaSuccess) {
                c->graph = nullptr;
                return cuda_err3(c, e, "cudaGraphInstantiate");
            }
        }
        for (; left >= kLen; left -= kLen) {
            cudaError_t e = cudaGraphLaunch(c->graph, c->stream);
            if (e != cudaSuccess) return cuda_err3(c, e, "cudaGraphLaunch");
        }
    }
    for (; left > 0; --left)
        if (step_once(c)) return cuda_err3(c, cudaGetLastError(), "step launch");
    c->step += n;
    return LBM_OK;
}

int lbm3d_get_fields(lbm3d_ctx* c, double* rho, double* ux, double* uy, double* uz, double* T) {
    if (!c) return LBM_EINVAL;
    if (!c->initialized) return set_err3(c, LBM_ESTATE, "no state yet");
    int rc = export_fields(c, 0);
    if (rc) return rc;
    const size_t N = (size_t)c->nx * c->ny * c->nz;
    double* dst[5] = {rho, ux, uy, uz, T};
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 5 && e == cudaSuccess; ++k)
        if (dst[k])
            e = cudaMemcpyAsync(dst[k], c->host_buf + k * N, N * sizeof(double), cudaMemcpyDeviceToHost,
                                c->stream);
    if (e != cudaSuccess) return cuda_err3(c, e, "copying fields to the host");
    return check3(c);
}

int lbm3d_get_populations(lbm3d_ctx* c, double* f, double* g, double* P) {
    if (!c) return LBM_EINVAL;
    if (!c->initialized) return set_err3(c, LBM_ESTATE, "no state yet");
    int rc = ensure_buf(c);
    if (rc) return rc;
    const size_t N = (size_t)c->nx * c->ny * c->nz;
    const dim3 b = blk3(), gr = grd3(c);
    if (c->prec == LBM_FP64)
        k3_export<double><<<gr, b, 0, c->stream>>>(c->D, make_lat3<double>(c->params, c->D), 1, c->host_buf);
    else
        k3_export<float><<<gr, b, 0, c->stream>>>(c->D, make_lat3<float>(c->params, c->D), 1, c->host_buf);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && f)
        e = cudaMemcpyAsync(f, c->host_buf, 19 * N * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && g)
        e = cudaMemcpyAsync(g, c->host_buf + 19 * N, 7 * N * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && P)
        e = cudaMemcpyAsync(P, c->host_buf + 26 * N, N * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e != cudaSuccess) return cuda_err3(c, e, "copying populations to the host");
    return check_state(c);
}

int lbm3d_diagnostics(lbm3d_ctx* c, double rho_l, double rho_g, int sessile, lbm_diag* out) {
    if (!c || !out || !(rho_l > rho_g)) return LBM_EINVAL;
    if (!c->initialized) return set_err3(c, LBM_ESTATE, "no state yet");
    int rc = export_fields(c, 2);
    if (rc) return rc;
    const size_t N = (size_t)c->nx * c->ny * c->nz;
    // the reduction takes |u| in place of u_x and zeros for u_y
    if (diag_launch(c->host_buf, c->host_buf + 5 * N, c->zeros, c->host_buf + 4 * N, (long long)N,
                    c->params.cv, rho_l, rho_g, c->diag_out, c->diag_scratch, c->stream))
        return cuda_err3(c, cudaGetLastError(), "diagnostics kernel");
    double h[8];
    cudaError_t e = cudaMemcpyAsync(h, c->diag_out, 7 * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_err3(c, e, "diagnostics");
    out->mass = h[0];
    out->energy = h[1];
    out->liquid_mass = h[2];
    out->liquid_area = h[3];
    out->liquid_area_smooth = h[4];
    out->max_u = h[5];
    out->nonfinite = (int)h[6];
    const double fac = sessile ? 12.0 / M_PI : 6.0 / M_PI;
    out->diameter = cbrt(fac * out->liquid_area);
    out->diameter_smooth = cbrt(fac * out->liquid_area_smooth);
    out->step = c->step;
    return check3(c);
}

long long lbm3d_step_count(const lbm3d_ctx* c) { return c ? c->step : -1; }

int lbm3d_set_path(lbm3d_ctx* c, int fused, int zseg) {
    if (!c || zseg < 0) return LBM_EINVAL;
    const bool f = fused != 0;
    const int zs = zseg == 0 ? auto_zseg(c->nx, c->ny, c->nz, c->prec) : (zseg > c->nz ? c->nz : zseg);
    if (f != c->fused || zs != c->zseg) {
        if (c->graph) cudaGraphExecDestroy(c->graph);
        c->graph = nullptr;
    }
    c->fused = f;
    c->zseg = zs;
    return LBM_OK;
}

int lbm3d_get_path(const lbm3d_ctx* c, int* fused, int* zseg) {
    if (!c) return LBM_EINVAL;
    if (fused) *fused = c->fused ? 1 : 0;
    if (zseg) *zseg = c->zseg;
    return LBM_OK;
}

int lbm3d_sync(lbm3d_ctx* c) {
    if (!c) return LBM_EINVAL;
    if (!c->initialized) return LBM_OK;
    return check_state(c);
}

void lbm3d_destroy(lbm3d_ctx* c) {
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    if (c->graph) cudaGraphExecDestroy(c->graph);
    if (c->host_buf) cudaFree(c->host_buf);
    if (c->diag_scratch) cudaFree(c->diag_scratch);
    if (c->diag_out) cudaFree(c->diag_out);
    if (c->zeros) cudaFree(c->zeros);
    if (c->mem) cudaFree(c->mem);
    if (c->ctl) cudaFree(c->ctl);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
    delete c;
}

const char* lbm3d_last_error(const lbm3d_ctx* c) { return c ? c->err.c_str() : "null context"; }

}  // extern "C"
