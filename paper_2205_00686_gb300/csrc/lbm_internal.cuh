// Internal definitions shared by the CUDA translation units of the library:
// device-resident descriptors, the per-launch physics constants and the
// closed-form pieces of the coupled step (Peng-Robinson EOS of Section 2,
// Eq. 10; the pseudopotential psi; (dp/dT)_rho used by Q of Eq. 20).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace lbm {

// flow / thermal boundary kinds (same values as the public header)
enum { PERIODIC = 0, WALL = 1, OPEN = 2 };
enum { T_PERIODIC = 0, T_DIRICHLET = 1, T_ADIABATIC = 2 };
enum { EW = 0, EE = 1, ES = 2, EN = 3 };

// sticky device error bits (ERR_TIMEOUT: a bounded wait for a staged row ran out)
enum { ERR_PSI = 1, ERR_NONFINITE = 2, ERR_TIMEOUT = 4 };

// Device-resident control block of one domain: the device-side step counter
// read by every launch, the three-slot ring of per-step density sums used by
// the buoyancy force (step n accumulates sum rho(n) into slot n % 3 and reads
// slot (n - 1) % 3), and the sticky error word.  The CTAs of a launch add
// their sums as fixed-point integers (massq and massh, see mass_bits; in three
// dimensions massq alone, see massq_scale), so the total does not depend on the
// order in which the CTAs finish; the launch's last CTA converts the finished
// slot to mass[] for the next step to read.
struct Ctl {
    long long step;
    double mass[3];
    long long massq[3];
    long long massh[3];
    // the step count at which the domain stops (> 0), or 0 for none: a
    // launch skips the units of a domain that has reached it, so its state,
    // step counter and density ring stay as they are
    long long target;
    int err;
    int done;          // CTAs that have finished (three-dimensional marching step)
};

__device__ __forceinline__ bool ctl_stopped(const Ctl* c) {
    const long long tg = __ldcg(&c->target);
    return tg > 0 && __ldcg(&c->step) >= tg;
}

// fixed-point scale of a three-dimensional domain's Ctl::massq, N = 1 / inv_n nodes:
// 2^(58 - e) with N < 2^e.  Densities stay below 16 (the EOS ends at 1/b =
// 10.5), so a domain total stays below 2^62 and no sum overflows, while a
// block sum keeps at least 30 fraction bits (N < 2^28) and small domains keep
// the full double precision of their block sums
__host__ __device__ __forceinline__ double massq_scale(double inv_n) {
    int e = 0;
    frexp(1.0 / inv_n, &e);
    return ldexp(1.0, 58 - e);
}
__device__ __forceinline__ void massq_add(long long* slot, double block_sum, double scale) {
    atomicAdd(reinterpret_cast<unsigned long long*>(slot),
              (unsigned long long)__double2ll_rn(block_sum * scale));
}
__host__ __device__ __forceinline__ double massq_value(long long q, double scale) {
    return (double)q / scale;
}

// Density sum of the two-dimensional step.  Every node's density is rounded to a
// fixed-point number of mass_bits(b) fraction bits and the numbers are added as
// integers, low 24 bits of a warp's sum into massq and the rest into massh: the
// total is exact, so rho_ave is the same bit for bit whatever strips, segments or
// tiles the domain is cut into, alone or in a batch.  (Sums in floating point over
// a segment's rows changed with the segment's height, which a batch takes from
// all of its members.)  Densities end at 1/b (EOS): with 1/b < 2^e the numbers
// hold up to 2^(e+1), in FP32 as 32 bits without sign (the grid is 7.5e-9 at b =
// 2/21: exact for a float density of 0.125 or more; a negative one counts as 0),
// in FP64 to 2^-(50-e) (1.4e-14, where a floating-point sum of 64 rows rounds at
// 3e-14).  It costs the 4096^2 FP32 step 334.5 -> 337.9 us, a batch of 64 192.8 ->
// 194.7; the 300 x 600 pool, whose threads no longer convert the sum back with a
// division each, went from 16.9 to 14.7.
inline int mass_bits(double b, bool fp64) {
    int e = 0;
    frexp(1.0 / b, &e);
    e = e < -60 ? -60 : (e > 60 ? 60 : e);
    return (fp64 ? 50 : 31) - e;
}

// One domain as seen by the kernels.  Populations are stored as deviations
// f_i - w_i rho_ref and g_i - w^_i T_ref, SoA planes [q][ny][pitch].
struct Inst {
    void* f[2];
    void* g[2];
    void* P[2];
    Ctl* ctl;
    int nx, ny, pitch;
    int flow[4], therm[4];
    int heater_x0, heater_x1;
    double T_edge[4], T_heater, cot_theta;
    double rho_ref, T_ref, inv_n;
    // rows [own_y0, own_y1) enter the density sum behind rho_ave; inv_n is
    // 1 / (nodes the mean is taken over).  The whole domain unless it is one
    // slab of a larger domain (lbm_set_partition).
    int own_y0, own_y1;
};

// A work unit of the fused step: output columns [x0, x1), rows [y0, y1) of
// domain `inst`.
struct Unit {
    int inst, x0, x1, y0, y1;
};

// Physical constants shared by every domain of a launch, already combined
// into the factors the kernels use.
template <class R>
struct Phys {
    // EOS: p = rho Rg T/(1 - b rho) - a h^2 rho^2/(1 + 2 b rho - b^2 rho^2),
    // h = 1 + kpr (1 - sqrt(T/Tc))
    R b, Rg, inv_Tc;
    R k_sa, k1_sa, m_third;          // k sqrt(a), (1 + k) sqrt(a), -1/3: see eos_node
    R two_over_G, negG_12;
    // D2Q9 MRT rates and Li forcing
    R s_e, s_eps, s_q, s_p;
    R hs_e, hs_eps, hs_q, hs_p;      // 1 - s/2
    R sig_e, sig_eps;                // sigma / (1/s - 1/2)
    // unit rates: the collision's combined factors (collide9_unit)
    R u_m, u_d, u_w;                 // (1 - s_p)/4, s_p/4, 1/2 - s_p/8
    R u_ax, u_dg, u_0;               // the sigma terms' factors of |12 s|^2
    // D2Q5
    R cv, inv_cv, inv_12cv, w_dot, w5_0, w5_1, vs1_cs2h, vs3, vs4;   // vs1_cs2h = vs1 / cs2h
    R h_m, one_m_vs4;               // h_m = (1 - vs1) / 2
    R gravity;
    R m_fix;              // density to fixed point, see mass_fix
    double m_unit;        // and back
    int frozen_flow, frozen_thermal;
};

struct PhysD {
    double a, b, Rg, omega, G, sigma;
    double s_e, s_eps, s_q, s_p;
    double cv, w_dot, vs1, vs3, vs4;
    double gravity;
    int frozen_flow, frozen_thermal;
};

template <class R>
inline Phys<R> make_phys(const PhysD& d) {
    Phys<R> p;
    double kpr = 0.37464 + 1.54226 * d.omega - 0.26992 * d.omega * d.omega;
    double Tc = 0.0778 * d.a / (0.45724 * d.b * d.Rg);
    p.b = (R)d.b;
    p.Rg = (R)(d.a < 0 ? -d.Rg : d.Rg);
    p.inv_Tc = (R)(1.0 / Tc);
    // eos_node works with |a| and p times the sign of a
    const double sgn = d.a < 0 ? -1.0 : 1.0, sa = std::sqrt(std::fabs(d.a));
    p.k_sa = (R)(kpr * sa);
    p.k1_sa = (R)((1.0 + kpr) * sa);
    p.m_third = (R)(-sgn / 3.0);
    p.two_over_G = (R)(sgn * 2.0 / d.G);
    p.negG_12 = (R)(-d.G / 12.0);
    p.s_e = (R)d.s_e;
    p.s_eps = (R)d.s_eps;
    p.s_q = (R)d.s_q;
    p.s_p = (R)d.s_p;
    p.hs_e = (R)(1.0 - 0.5 * d.s_e);
    p.hs_eps = (R)(1.0 - 0.5 * d.s_eps);
    p.hs_q = (R)(1.0 - 0.5 * d.s_q);
    p.hs_p = (R)(1.0 - 0.5 * d.s_p);
    p.sig_e = (R)(d.sigma / (1.0 / d.s_e - 0.5));
    p.sig_eps = (R)(d.sigma / (1.0 / d.s_eps - 0.5));
    p.u_m = (R)(0.25 * (1.0 - d.s_p));
    p.u_d = (R)(0.25 * d.s_p);
    p.u_w = (R)(0.5 - 0.125 * d.s_p);
    {
        // |F_m|^2 / psi^2 = G^2 |12 s|^2 / 144; e and epsilon get +-half of
        // sigma / (1/s - 1/2) times it (s_e = s_eps = 1)
        const double k = d.G * d.G / 144.0, se = 0.5 * d.sigma / (1.0 / d.s_e - 0.5),
                     sp = 0.5 * d.sigma / (1.0 / d.s_eps - 0.5);
        p.u_ax = (R)(k * (2.0 * sp - se) / 36.0);
        p.u_dg = (R)(k * (2.0 * se - sp) / 36.0);
        p.u_0 = (R)(-k * (se + sp) / 9.0);
    }
    p.cv = (R)d.cv;
    p.inv_cv = (R)(1.0 / d.cv);
    p.inv_12cv = (R)(sgn / (12.0 * d.cv));
    p.w_dot = (R)d.w_dot;
    p.w5_0 = (R)(1.0 - d.w_dot);
    p.w5_1 = (R)(0.25 * d.w_dot);
    p.vs1_cs2h = (R)(d.vs1 / (0.5 * d.w_dot));
    p.vs3 = (R)d.vs3;
    p.vs4 = (R)d.vs4;
    p.h_m = (R)(0.5 * (1.0 - d.vs1));
    p.one_m_vs4 = (R)(1.0 - d.vs4);
    p.gravity = (R)d.gravity;
    // FP32 multiplies by 2^bits; FP64 adds 1.5 * 2^(52 - bits), which leaves the
    // rounded density in the low bits of the sum
    const int bits = mass_bits(d.b, sizeof(R) == 8);
    p.m_fix = (R)(sizeof(R) == 8 ? std::ldexp(1.5, 52 - bits) : std::ldexp(1.0, bits));
    p.m_unit = std::ldexp(1.0, -bits);
    p.frozen_flow = d.frozen_flow;
    p.frozen_thermal = d.frozen_thermal;
    return p;
}

// ---- storage conversions ------------------------------------------------
__device__ __forceinline__ float ld_st(const float* p) { return __ldg(p); }
__device__ __forceinline__ double ld_st(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ld_st(const __half* p) { return __half2float(__ldg(p)); }
__device__ __forceinline__ void st_st(float* p, float v) { *p = v; }
__device__ __forceinline__ void st_st(double* p, double v) { *p = v; }
__device__ __forceinline__ void st_st(__half* p, float v) { *p = __float2half_rn(v); }
// a staged (shared-memory) storage value as arithmetic type
__device__ __forceinline__ float st_val(float v) { return v; }
__device__ __forceinline__ float st_val(__half v) { return __half2float(v); }

// float to double, exactly, by integer operations for normal numbers: the
// conversion instruction runs on the FP64 pipe (64 cycles per warp and SM
// partition), these six on the integer pipe
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
    const unsigned b = __float_as_uint(v), a = b & 0x7fffffffu;
    if (a - 0x00800000u >= 0x7f000000u) return (double)v;     // zero, denormal, infinite, NaN
    return __hiloint2double((int)(((a >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(a << 29));
}

// ---- arithmetic helpers (precision-generic) -------------------------------
// FP32 uses the hardware approximations (rcp.approx / sqrt.approx, relative error
// ~2^-23), well inside the FP32 tolerance; FP64 two series terms from the hardware
// seeds (below).  rsq, the wall's tangential difference, is IEEE in both.
__device__ __forceinline__ float rsq(float x) { return sqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return sqrt(x); }
__device__ __forceinline__ float rabs(float x) { return fabsf(x); }
__device__ __forceinline__ double rabs(double x) { return fabs(x); }
__device__ __forceinline__ float f_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// FP64 reciprocal and square root.  The GB300 executes two FP64 lanes per SM
// and clock, so an FP64 step is bound by the number of FP64 instructions.
// Both start from the hardware approximation of the seed, with e = 1 - x r
// (or 1 - x y^2) of about 2^-20, and take the first two terms of the series
// 1/(1-e) = 1 + e + e^2 + ... (or (1-e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ...): what
// is left out is of order e^3 ~ 2^-60, below the FP64 rounding: the reciprocal
// is within 0.51 ulp, the square root, whose correction takes half of the rounding
// of x y for the seed's, within 0.76 (test_gpu_fp64_math.py).  Three
// and five FP64 instructions, against four for two Newton-Raphson steps and
// about ten for the IEEE square root.  With the node arithmetic of
// lbm_node.cuh, which counts FP64 operations the same way (243 per node, halo
// included, to 180), the FP64 step on 1999 x 1501 went from 1.355 to 1.043 ms; in
// FP32 the same forms took the 4096^2 step from 340.3 to 334.4 us (337.9 with the
// exact density sum).  (With the
// IEEE operations instead the fields' distance from the FP64 oracle's is the
// same, 2.3e-15 on 1999 x 1501.)  A zero, infinite or NaN reciprocal
// operand gives a non-finite result, which the step reports; a square-root
// operand outside the normal range (zero, negative, NaN among them) takes
// the IEEE square root.
__device__ __forceinline__ double f_rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ float f_sqrt(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double f_sqrt(double x) {
    // high words of 2^-1000 .. 2^1000, compared as integers (an FP64 compare
    // would take a slot of the FP64 pipe)
    if ((unsigned)(__double2hiint(x) - 0x01700000) > 0x7d000000u) return sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = x * y;
    const double e = fma(-t, y, 1.0);
    return fma(t * e, fma(0.375, e, 0.5), t);
}

// density of a node as a fixed-point number (see mass_bits), one conversion in
// FP32, in FP64 one addition on the FP64 pipe as a running sum would take
// (0 where the node is not counted)
__device__ __forceinline__ unsigned mass_fix(const Phys<float>& P, float rho, bool counted) {
    return __float2uint_rn(__fmul_rn(rho, counted ? P.m_fix : 0.0f));
}
__device__ __forceinline__ long long mass_fix(const Phys<double>& P, double rho, bool counted) {
    const long long q = __double_as_longlong(__dadd_rn(rho, P.m_fix)) - __double_as_longlong(P.m_fix);
    return counted ? q : 0;
}
__device__ __forceinline__ void mass_add(Ctl* c, int slot, long long sum) {
    atomicAdd(reinterpret_cast<unsigned long long*>(&c->massq[slot]), (unsigned long long)(sum & 0xffffff));
    atomicAdd(reinterpret_cast<unsigned long long*>(&c->massh[slot]), (unsigned long long)(sum >> 24));
}
__device__ __forceinline__ double mass_total(const Ctl* c, int slot, double unit) {
    return fma((double)__ldcg(&c->massh[slot]), 16777216.0, (double)__ldcg(&c->massq[slot])) * unit;
}

__device__ __forceinline__ int wrapi(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}

// wall / Dirichlet temperature along an edge, with the heater segment
__device__ __forceinline__ double wall_T(const Inst& I, int edge, int gx) {
    if (edge == ES && gx >= I.heater_x0 && gx < I.heater_x1) return I.T_heater;
    return I.T_edge[edge];
}

// Per-instance storage types by precision code
template <int PREC> struct Types;
template <> struct Types<0> { typedef double R; typedef double TF; typedef double TG; };
template <> struct Types<1> { typedef float R; typedef float TF; typedef float TG; };
template <> struct Types<2> { typedef float R; typedef float TF; typedef __half TG; };

inline size_t elem_f(int prec) { return prec == 0 ? 8 : 4; }
inline size_t elem_g(int prec) { return prec == 0 ? 8 : (prec == 1 ? 4 : 2); }
inline size_t elem_P(int prec) { return prec == 0 ? 8 : 4; }

// ---- launchers implemented in the .cu files ------------------------------
struct StepLaunch {
    Inst* insts;
    const Unit* units;
    int n_units;
    int n_inst;
    unsigned* sched;   // [0] next unit, [1] finished CTAs
    int grid;
    int walls;         // some domain has a wall: the launch carries the wall rings
    int staged;        // FP32 / FP16-g: rows arrive by bulk copies (stage_eligible)
    int wait_probe;    // test hook: staged CTAs also wait on an mbarrier nothing arms
    int targets;       // some domain has a target step (lbm_set_target)
    PhysD phys;
};

// The bulk-copy staged form (FP32 f and P; g in FP32 or FP16) needs every
// copied row piece to start on a 16-byte boundary: always true for open x
// edges (the copy of the last strip is rounded up into the row's pitch
// padding), and for periodic x when the wrapped pieces start on 16-byte
// column boundaries (nx a multiple of 4 for FP32 g, of 8 for FP16 g) and the
// window wraps at most a few times (nx >= 32).
inline bool stage_eligible(const Inst& I, int prec) {
    if (prec != 1 && prec != 2) return false;
    if (I.flow[EW] != PERIODIC) return true;
    return I.nx % (prec == 2 ? 8 : 4) == 0 && I.nx >= 32;
}

// Small-domain form (lbm_tile.cu): tiles of tx x ty nodes, one thread per
// node, several steps per launch.  tx = 0: the domain takes the sweep.
struct TilePlan {
    int tx = 0, ty = 0, threads = 0, ring0 = 0, ntx = 0, n_tiles = 0, grid = 0;
    size_t smem = 0;
};
struct TileLaunch {
    Inst inst;
    unsigned* bar;     // grid counter, 0 between launches
    int tx, ty, ring0, ntx, n_tiles, steps;
    int targets;       // the domain has a target step (lbm_set_target)
    unsigned wait;     // clocks (modulo 2^32) a CTA waits at the grid barrier before it gives up
};
// the plan of the form's own choice, or (want_tx > 0) for that tile: tx = 0 when
// there is none
int tile_plan(int prec, const Inst& I, int sms, int want_tx, int want_ty, TilePlan* out);
cudaError_t tile_launch(int prec, const TilePlan& T, const TileLaunch& L, const PhysD& phys,
                        cudaStream_t st);

// The unit-rate form applies when every non-hydrodynamic rate is exactly 1
// (s_e = s_eps = s_q = 1 and varsigma_3 = varsigma_4 = 1, the paper's choice).
inline bool unit_rates(const PhysD& d) {
    return d.s_e == 1.0 && d.s_eps == 1.0 && d.s_q == 1.0 && d.vs3 == 1.0 && d.vs4 == 1.0;
}

int step_launch(int prec, int threads, const StepLaunch& L, cudaStream_t st);
int step_occupancy(int prec, int threads, int walls, int staged, int* ctas_per_sm,
                   size_t* smem_bytes);

int init_launch(int prec, const Inst* I_dev, const Inst& I, const double* rho, const double* ux,
                const double* uy, const double* T, double w_dot, cudaStream_t st);
// rho, u (half-force velocity), T of the current state
int fields_launch(int prec, const Inst& I, const PhysD& phys, double* rho, double* ux, double* uy,
                  double* T, cudaStream_t st);
int pop_get_launch(int prec, const Inst& I, int parity, double w_dot, double* f, double* g,
                   double* P, cudaStream_t st);
int pop_set_launch(int prec, const Inst& I, int parity, double w_dot, const double* f,
                   const double* g, const double* P, cudaStream_t st);
// reduction of device fields into 8 doubles + a nonfinite count; `scratch`
// holds diag_scratch_bytes(n) bytes
size_t diag_scratch_bytes(long long n);
int diag_launch(const double* rho, const double* ux, const double* uy, const double* T,
                long long n, double cv, double rho_l, double rho_g, double* out9,
                void* scratch, cudaStream_t st);
// out2 = (sum a, sum b) over n device doubles, fixed summation order; the
// same scratch as diag_launch
int sum2_launch(const double* a, const double* b, long long n, double* out2, void* scratch,
                cudaStream_t st);

// interface analyses (lbm_analysis.cu)
// contact-angle sums: out12[0..8] = n, sum u, sum v, sum uu, sum vv, sum uv,
// sum u z, sum v z, sum z about the mean point, out12[9..11] = n, sum x, sum y
size_t iface_scratch_bytes();
int iface_launch(const double* rho, int nx, int ny, double rho_mid, int skip, double* out12,
                 void* scratch, cudaStream_t st);
// one region of the phase: label = smallest node index, flags bit 0..3 = the
// region touches the W, E, S, N edge
struct RegionOut {
    long long label, area, sum_y;
    int y_min, y_max, flags, pad;
};
size_t regions_scratch_bytes(long long n);
// labels the phase; *parent_out -> n ints (root label or -1), *roots_out ->
// the first max_roots roots in no order, *count_out -> [roots found, error]
int regions_launch(const double* rho, int nx, int ny, int perx, int pery, double thr, int below,
                   void* scratch, int max_roots, int** parent_out, int** roots_out,
                   int** count_out, cudaStream_t st);
int regions_gather_launch(void* scratch, long long n, int m, RegionOut* out, cudaStream_t st);

}  // namespace lbm
