// Auxiliary kernels around the fused step: initial equilibrium populations,
// macroscopic fields of the current state (rho, u with the half-force
// correction of Eq. 11, T), population import / export as absolute doubles,
// and the FP64 diagnostics reduction.  None of these is on the per-step path.
#include <algorithm>

#include "lbm_node.cuh"

namespace lbm {

__constant__ int dCX9[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
__constant__ int dCY9[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
__constant__ double dW9[9] = {4.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9,
                              1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};

__device__ __forceinline__ double w5(int i, double w_dot) { return i == 0 ? 1.0 - w_dot : 0.25 * w_dot; }

// ---------------------------------------------------------------------------
// f = f^eq(rho, u) (Eq. 3), g = w^ T (Eq. 22), P = 0, stored as deviations
template <int PREC>
__global__ void k_init(Inst I, const double* rho, const double* ux, const double* uy,
                       const double* T, double w_dot) {
    typedef typename Types<PREC>::TF TF;
    typedef typename Types<PREC>::TG TG;
    typedef typename Types<PREC>::R R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= I.nx) return;
    const size_t n = (size_t)y * I.nx + x;
    const size_t plane = (size_t)I.ny * I.pitch;
    const size_t off = (size_t)y * I.pitch + x;
    const double r = rho[n], vx = ux[n], vy = uy[n], t = T[n];
    TF* f = (TF*)I.f[0];
    TG* g = (TG*)I.g[0];
    R* P = (R*)I.P[0];
    if (PREC == 0) {
        const double uu = vx * vx + vy * vy;
        for (int i = 0; i < 9; ++i) {
            const double cu = dCX9[i] * vx + dCY9[i] * vy;
            const double fe = dW9[i] * r * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
            st_st(f + i * plane + off, (TF)(fe - dW9[i] * I.rho_ref));
        }
        for (int i = 0; i < 5; ++i) st_st(g + i * plane + off, (R)(w5(i, w_dot) * (t - I.T_ref)));
    } else {
        // FP32 state: the deviation f^eq - w rho_ref = w [(rho - rho_ref) +
        // rho (3 c.u + 9/2 (c.u)^2 - 3/2 u^2)] in float (the reference
        // difference in double), which stays within the state's own rounding
        const float dr = (float)(r - I.rho_ref), rf = (float)r;
        const float fx = (float)vx, fy = (float)vy, uu = fx * fx + fy * fy;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const float cu = (float)dCX9[i] * fx + (float)dCY9[i] * fy;
            const float w = (float)dW9[i];
            st_st(f + i * plane + off, (TF)(w * (dr + rf * (3.0f * cu + 4.5f * cu * cu - 1.5f * uu))));
        }
        const float td = (float)(t - I.T_ref);
#pragma unroll
        for (int i = 0; i < 5; ++i) st_st(g + i * plane + off, (float)w5(i, w_dot) * td);
    }
    P[off] = R(0);
}

int init_launch(int prec, const Inst* I_dev, const Inst& I, const double* rho, const double* ux,
                const double* uy, const double* T, double w_dot, cudaStream_t st) {
    (void)I_dev;
    dim3 blk(128), grd((I.nx + 127) / 128, I.ny);
    if (prec == 0) k_init<0><<<grd, blk, 0, st>>>(I, rho, ux, uy, T, w_dot);
    else if (prec == 1) k_init<1><<<grd, blk, 0, st>>>(I, rho, ux, uy, T, w_dot);
    else k_init<2><<<grd, blk, 0, st>>>(I, rho, ux, uy, T, w_dot);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// Fields of the current state: rho, T and u = (j + F/2) / rho (Eq. 11) with F_m
// from the psi stencil (Eq. 9, wetting ghost layer of Section 3.3) and buoyancy,
// in the state's own precision, written as doubles.  A CTA takes 32 x 8 nodes;
// moments and psi of the tile and one node around it come from the populations
// (1.33 times the tile's), psi passes through shared memory.  Bound by memory:
// 56 B read and 32 B written per node (FP32).  One pass instead of two over five
// double fields, and float to double by integer operations (the conversion
// instruction runs on the FP64 pipe): 2048^2 FP32 200 -> 84 us.
constexpr int FTX = 32, FTY = 8;
template <int PREC>
__global__ void __launch_bounds__(FTX* FTY)
k_fields(const __grid_constant__ Inst I, const __grid_constant__ Phys<typename Types<PREC>::R> P,
         double* __restrict__ orho, double* __restrict__ oux, double* __restrict__ ouy,
         double* __restrict__ oT) {
    typedef typename Types<PREC>::R R;
    typedef typename Types<PREC>::TF TF;
    typedef typename Types<PREC>::TG TG;
    typedef typename Vec2<R>::T R2;
    constexpr int W = FTX + 2;
    __shared__ R s_psi[W * (FTY + 2)];
    const int nx = I.nx, ny = I.ny, t = threadIdx.x;
    const unsigned ntx = (nx + FTX - 1) / FTX;
    const int x0 = (int)(blockIdx.x % ntx) * FTX, y0 = (int)(blockIdx.x / ntx) * FTY;
    const long long step = __ldcg(&I.ctl->step);
    const int par = (int)(step & 1);
    const TF* const f = (const TF*)I.f[par];
    const TG* const g = (const TG*)I.g[par];
    const size_t plane = (size_t)ny * I.pitch;
    const bool perx = I.flow[EW] == PERIODIC, pery = I.flow[ES] == PERIODIC;
    const R rho_ref = (R)I.rho_ref, T_ref = (R)I.T_ref;
    auto load = [&](int x, int y, R* fv, R* gv) {
        const size_t off = (size_t)y * I.pitch + x;
#pragma unroll
        for (int q = 0; q < 9; ++q) fv[q] = (R)ld_st(f + q * plane + off);
#pragma unroll
        for (int q = 0; q < 5; ++q) gv[q] = (R)ld_st(g + q * plane + off);
    };
    int err = 0;     // the step reports errors; the read-out does not
    const int lx = t % FTX, ly = t / FTX, gx = x0 + lx, gy = y0 + ly;
    const int tw = min(FTX, nx - x0), th = min(FTY, ny - y0);
    const bool own = lx < tw && ly < th;
    const int c = (ly + 1) * W + lx + 1;
    Node<R> n;
    if (own) {
        R fv[9], gv[5];
        load(gx, gy, fv, gv);
        node_fields(P, rho_ref, T_ref, fv, gv, n);
        s_psi[c] = n.psi;
    }
    if (t < 2 * (tw + th) + 4) {
        // the ring around the tile: inside the domain (wrapped along periodic
        // axes), the ghost layer of a wall, or unused
        const int w = tw + 2;
        int rx, ry;
        if (t < w) { rx = t - 1; ry = -1; }
        else if (t < 2 * w) { rx = t - w - 1; ry = th; }
        else if (t < 2 * w + th) { rx = -1; ry = t - 2 * w; }
        else { rx = tw; ry = t - 2 * w - th; }
        const int r = (ry + 1) * W + rx + 1;
        int x = x0 + rx, y = y0 + ry;
        if (perx) x = wrapi(x, nx);
        if (pery) y = wrapi(y, ny);
        if (x >= 0 && x < nx) {
            R fv[9], gv[5];
            if (y >= 0 && y < ny) {
                Node<R> m;
                load(x, y, fv, gv);
                node_fields(P, rho_ref, T_ref, fv, gv, m);
                s_psi[r] = m.psi;
            } else if (I.flow[y < 0 ? ES : EN] == WALL) {
                const int y1 = y < 0 ? 0 : ny - 1, y2 = y < 0 ? 1 : ny - 2;
                const int xp = perx ? wrapi(x + 1, nx) : min(x + 1, nx - 1);
                const int xm = perx ? wrapi(x - 1, nx) : max(x - 1, 0);
                auto rho_at = [&](int xx, int yy) {
                    load(xx, yy, fv, gv);
                    return radd(sum9(fv), rho_ref);
                };
                const R rp = rho_at(xp, y1), rm = rho_at(xm, y1), far = rho_at(x, y2);
                load(x, y1, fv, gv);
                s_psi[r] = ghost_psi(P, far, rp, rm, (R)I.cot_theta, radd(sum5(gv), T_ref), &err);
            }
        }
    }
    __syncthreads();
    if (!own) return;
    const int dw = (!perx && gx == 0) ? 0 : -1, de = (!perx && gx == nx - 1) ? 0 : 1;
    const int ds = (I.flow[ES] == OPEN && gy == 0) ? 0 : -W, dn = (I.flow[EN] == OPEN && gy == ny - 1) ? 0 : W;
    const R* const p = s_psi + c;
    const R2 s12 = force_stencil<R>(p[dw], p[de], p[ds + dw], p[ds], p[ds + de], p[dn + dw], p[dn], p[dn + de]);
    R rho_ave = R(0);
    if (P.gravity != R(0)) rho_ave = (R)(__ldcg(&I.ctl->mass[(step + 2) % 3]) * I.inv_n);
    const R2 F = force_of<R>(P, s12, n.psi, n.rho, rho_ave);
    R ux = R(0), uy = R(0);
    if (!P.frozen_flow) {
        if constexpr (sizeof(R) == 8) {
            const R2 u = velocity<R>(F, pr(n.jx, n.jy), n.ir);
            ux = u.x;
            uy = u.y;
        } else {
            ux = __fdiv_rn(rfma(F.x, R(0.5), n.jx), n.rho);
            uy = __fdiv_rn(rfma(F.y, R(0.5), n.jy), n.rho);
        }
    }
    const size_t o = (size_t)gy * nx + gx;
    orho[o] = widen(n.rho);
    oux[o] = widen(ux);
    ouy[o] = widen(uy);
    oT[o] = widen(n.T);
}

int fields_launch(int prec, const Inst& I, const PhysD& phys, double* rho, double* ux, double* uy,
                  double* T, cudaStream_t st) {
    const unsigned grd = (unsigned)((I.nx + FTX - 1) / FTX) * (unsigned)((I.ny + FTY - 1) / FTY);
    if (prec == 0) k_fields<0><<<grd, FTX * FTY, 0, st>>>(I, make_phys<double>(phys), rho, ux, uy, T);
    else if (prec == 1) k_fields<1><<<grd, FTX * FTY, 0, st>>>(I, make_phys<float>(phys), rho, ux, uy, T);
    else k_fields<2><<<grd, FTX * FTY, 0, st>>>(I, make_phys<float>(phys), rho, ux, uy, T);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// populations as absolute doubles, [q][ny][nx]
template <int PREC>
__global__ void k_pop(Inst I, int par, double w_dot, double* f, double* g, double* P, int set) {
    typedef typename Types<PREC>::TF TF;
    typedef typename Types<PREC>::TG TG;
    typedef typename Types<PREC>::R R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= I.nx) return;
    const size_t plane = (size_t)I.ny * I.pitch, off = (size_t)y * I.pitch + x;
    const size_t dplane = (size_t)I.ny * I.nx, doff = (size_t)y * I.nx + x;
    TF* fs = (TF*)I.f[par];
    TG* gs = (TG*)I.g[par];
    R* Ps = (R*)I.P[par];
    if (set) {
        for (int i = 0; i < 9; ++i)
            st_st(fs + i * plane + off, (TF)(f[i * dplane + doff] - dW9[i] * I.rho_ref));
        for (int i = 0; i < 5; ++i)
            st_st(gs + i * plane + off, (R)(g[i * dplane + doff] - w5(i, w_dot) * I.T_ref));
        Ps[off] = (R)P[doff];
    } else {
        if (f)
            for (int i = 0; i < 9; ++i)
                f[i * dplane + doff] = (double)fs[i * plane + off] + dW9[i] * I.rho_ref;
        if (g)
            for (int i = 0; i < 5; ++i)
                g[i * dplane + doff] = (double)ld_st(gs + i * plane + off) + w5(i, w_dot) * I.T_ref;
        if (P) P[doff] = (double)Ps[off];
    }
}

static int pop_launch(int prec, const Inst& I, int par, double w_dot, double* f, double* g,
                      double* P, int set, cudaStream_t st) {
    dim3 blk(128), grd((I.nx + 127) / 128, I.ny);
    if (prec == 0) k_pop<0><<<grd, blk, 0, st>>>(I, par, w_dot, f, g, P, set);
    else if (prec == 1) k_pop<1><<<grd, blk, 0, st>>>(I, par, w_dot, f, g, P, set);
    else k_pop<2><<<grd, blk, 0, st>>>(I, par, w_dot, f, g, P, set);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int pop_get_launch(int prec, const Inst& I, int par, double w_dot, double* f, double* g,
                   double* P, cudaStream_t st) {
    return pop_launch(prec, I, par, w_dot, f, g, P, 0, st);
}

int pop_set_launch(int prec, const Inst& I, int par, double w_dot, const double* f,
                   const double* g, const double* P, cudaStream_t st) {
    return pop_launch(prec, I, par, w_dot, (double*)f, (double*)g, (double*)P, 1, st);
}

// ---------------------------------------------------------------------------
// diagnostics: per-block partial sums in double, then the last block to finish
// folds the partials, one warp per value, in a fixed order (deterministic
// result).  Bound by the FP64 pipe: 13 FP64 operations per node (no division, no
// square root per node, finiteness by integer tests).  2048^2 308 -> 114 us; small
// fields take fewer blocks, whose fold is what they wait for.
enum { DIAG_BLOCKS = 304, DIAG_THREADS = 256, DIAG_VALS = 7 };
inline int diag_blocks(long long n) {
    return (int)std::min<long long>(DIAG_BLOCKS, std::max<long long>(1, (n + 2 * DIAG_THREADS - 1) / (2 * DIAG_THREADS)));
}

__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// folds n_vals values of n_blocks partials ([block][value]) by warps: lane l adds
// blocks l, l + 32, ... in order, then the lanes pairwise; value `vmax` (if any)
// by maximum.  All threads of the block take part; fin(k, v) in lane 0.
template <class Fin>
__device__ __forceinline__ void fold_partials(const double* partial, unsigned n_blocks, int n_vals, int vmax,
                                              Fin fin) {
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < n_vals; k += blockDim.x >> 5) {
        double x = 0.0;
        for (unsigned b = lane; b < n_blocks; b += 32) {
            const double y = __ldcg(&partial[b * n_vals + k]);
            x = k == vmax ? fmax(x, y) : x + y;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double y = __shfl_down_sync(0xffffffffu, x, o);
            x = k == vmax ? fmax(x, y) : x + y;
        }
        if (lane == 0) fin(k, x);
    }
}

size_t diag_scratch_bytes(long long n) {
    (void)n;
    return (size_t)DIAG_BLOCKS * DIAG_VALS * sizeof(double) + 256;
}

__global__ void __launch_bounds__(DIAG_THREADS)
    k_diag(const double* rho, const double* ux, const double* uy, const double* T, long long n,
           double cv, double rho_l, double rho_g, double* out, double* partial,
           unsigned* ticket) {
    __shared__ double red[DIAG_VALS][DIAG_THREADS / 32];
    __shared__ bool last;
    const double rmid = 0.5 * (rho_l + rho_g), inv = 1.0 / (rho_l - rho_g);
    double v[DIAG_VALS] = {0, 0, 0, 0, 0, 0, 0};
    unsigned n_liq = 0, n_bad = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double r = rho[i], a = ux[i], b = uy[i], t = T[i];
        v[0] += r;
        v[1] += r * t;
        if (r > rmid) {
            v[2] += r;
            ++n_liq;
        }
        const double ph = (r - rho_g) * inv;
        v[4] += ph < 0.0 ? 0.0 : (ph > 1.0 ? 1.0 : ph);
        v[5] = fmax(v[5], fma(a, a, b * b));
        n_bad += finite(r) && finite(a) && finite(b) && finite(t) ? 0u : 1u;
    }
    v[1] *= cv;
    v[3] = (double)n_liq;
    v[5] = sqrt(v[5]);
    v[6] = (double)n_bad;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = 0; k < DIAG_VALS; ++k) {
        double x = v[k];
        for (int o = 16; o > 0; o >>= 1) {
            const double y = __shfl_down_sync(0xffffffffu, x, o);
            x = k == 5 ? fmax(x, y) : x + y;
        }
        if (lane == 0) red[k][wid] = x;
    }
    __syncthreads();
    if (threadIdx.x < DIAG_VALS) {
        const int k = threadIdx.x;
        double x = red[k][0];
        for (int w = 1; w < DIAG_THREADS / 32; ++w) x = k == 5 ? fmax(x, red[k][w]) : x + red[k][w];
        partial[blockIdx.x * DIAG_VALS + k] = x;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) {
        __threadfence();
        fold_partials(partial, gridDim.x, DIAG_VALS, 5, [&](int k, double x) {
            out[k] = x;
            if (k == 0) *ticket = 0u;
        });
    }
}

// sum rho and sum T of device fields (the storage references and the first
// step's mean density), with the same fixed-order two-level reduction
__global__ void __launch_bounds__(DIAG_THREADS)
    k_sum2(const double* a, const double* b, long long n, double* out, double* partial,
           unsigned* ticket) {
    __shared__ double red[2][DIAG_THREADS / 32];
    __shared__ bool last;
    double v0 = 0.0, v1 = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        v0 += a[i];
        v1 += b[i];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_down_sync(0xffffffffu, v0, o);
        v1 += __shfl_down_sync(0xffffffffu, v1, o);
    }
    if (lane == 0) {
        red[0][wid] = v0;
        red[1][wid] = v1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const int k = threadIdx.x;
        double x = red[k][0];
        for (int w = 1; w < DIAG_THREADS / 32; ++w) x += red[k][w];
        partial[blockIdx.x * 2 + k] = x;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) {
        __threadfence();
        fold_partials(partial, gridDim.x, 2, -1, [&](int k, double x) {
            out[k] = x;
            if (k == 0) *ticket = 0u;
        });
    }
}

int sum2_launch(const double* a, const double* b, long long n, double* out2, void* scratch,
                cudaStream_t st) {
    double* partial = (double*)scratch;
    unsigned* ticket = (unsigned*)((char*)scratch + (size_t)DIAG_BLOCKS * DIAG_VALS * sizeof(double));
    k_sum2<<<diag_blocks(n), DIAG_THREADS, 0, st>>>(a, b, n, out2, partial, ticket);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int diag_launch(const double* rho, const double* ux, const double* uy, const double* T,
                long long n, double cv, double rho_l, double rho_g, double* out9, void* scratch,
                cudaStream_t st) {
    double* partial = (double*)scratch;
    unsigned* ticket = (unsigned*)((char*)scratch + (size_t)DIAG_BLOCKS * DIAG_VALS * sizeof(double));
    k_diag<<<diag_blocks(n), DIAG_THREADS, 0, st>>>(rho, ux, uy, T, n, cv, rho_l, rho_g, out9,
                                                 partial, ticket);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace lbm
