// Small-domain form of the coupled step: several time steps per launch, one
// two-dimensional tile of nodes per CTA, every node's thread kept for the
// whole launch.
//
// The sweep of lbm_step.cu is made for bandwidth: a CTA walks a strip row by
// row, so a step of a small domain is a chain of (rows + 6) iterations of two
// barriers each on the few CTAs the domain fills (64 x 64 in FP64: 14
// iterations on 8 of 152 SMs, 83 us).  Here the state stays in L2, a step of a
// tile is one pass of three stages, each closed by a barrier of the CTA, and the
// tile is small enough that the domain reaches all SMs:
//   A  moments, EOS and psi of the tile and two nodes around it (a thread loads
//      the 15 values of its node and the 14 of its node around the tile before
//      the first is used)
//   B  F_m, F, u on the tile and one node around it; on the tile the D2Q9
//      collision, f*_i pushed to its destination in f(t+1) (wall: back to this
//      node as the opposite direction; open edge: also to the edge nodes whose
//      source clamps to this node)
//   C  on the tile div u, Q, S, the D2Q5 collision; g*_i blended into its
//      destination's g(t+1) (Eq. 39; thermal walls return it to this node)
// Each node is collided once, by its owner; only moments and psi (two nodes
// around) and u (one node) are formed again by the neighbouring tiles.
//
// Steps of one launch are separated by a barrier over the grid (a counter in
// device memory; the launch is cooperative, so every CTA is resident).  The
// wait is bounded: after about a second a CTA records ERR_TIMEOUT and leaves, and
// the others with it.
// What a step reads that another CTA wrote goes through L2 (ld.global.cg).
// The arithmetic is that of lbm_node.cuh, so the state is bit for bit the one
// the sweep would give.
//
// Measured per step (one GB300, lbm_step of 60-300 steps, sweep -> this): FP32
// 64^2 18.1 -> 3.45 us, 256^2 18.5 -> 5.0, 300 x 600 pool 20.5 -> 12.8, 512^2
// 22.3 -> 14.9; FP16-g 400 x 200 with a wall 20.8 -> 7.7; FP64 64^2 82 -> 8.9,
// 200^2 87 -> 21.4, 384^2 149 -> 71.  512^2 FP32: 837 thread instructions per node
// (sweep 462), issue 40 % active, barriers the top stall.
#include <algorithm>

#include "lbm_node.cuh"

namespace lbm {

namespace {

template <class T>
__device__ __forceinline__ T ld_l2(const T* p) { return __ldcg(p); }
__device__ __forceinline__ float ld_l2(const __half* p) {
    return __half2float(__ushort_as_half(__ldcg(reinterpret_cast<const unsigned short*>(p))));
}

// Most threads per CTA.  FP32: up to 512, so that 128 registers are left (two CTAs
// of 256 threads per SM; at 80 registers three fit but spill: 300 x 600 15.3 ->
// 18.5 us per step, 256^2 5.1 -> 6.5).  FP64: up to 288 (20 x 14 nodes, 168
// registers), so that 200 x 200 fits one round of 152 SMs.
constexpr int TILE_MAX(int prec) { return prec == 0 ? 288 : 512; }

// Set in the grid counter by a CTA that gave up its wait: the others leave at
// their next look at the counter, and so do the launches queued behind this one,
// until lbm_init_fields, lbm_set_populations or lbm_load clears it.  (Counts stay
// below 1024 steps times a few thousand CTAs.)
constexpr unsigned BAR_LEFT = 1u << 30;

// release / acquire on the grid counter
__device__ __forceinline__ unsigned bar_load(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned bar_add(unsigned* p) {
    unsigned v;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// shared memory of a tile (element counts for tile + 2 and tile + 1 nodes)
__host__ __device__ inline size_t tile_bytes(size_t es, int tx, int ty) {
    const int n2 = (tx + 4) * (ty + 4), n1 = (tx + 2) * (ty + 2);
    return (size_t)(((n2 + 1) & ~1) + 7 * n1) * es;
}

template <int PREC, bool UNIT>
__global__ void __launch_bounds__(TILE_MAX(PREC))
k_tile(const __grid_constant__ TileLaunch L, const __grid_constant__ Phys<typename Types<PREC>::R> P) {
    typedef typename Types<PREC>::R R;
    typedef typename Types<PREC>::TF TF;
    typedef typename Types<PREC>::TG TG;
    typedef typename Vec2<R>::T R2;
    const Inst& I = L.inst;
    const int TX = L.tx, TY = L.ty, W2 = TX + 4, W1 = TX + 2;
    const int N2 = W2 * (TY + 4), N1 = W1 * (TY + 2);
    extern __shared__ __align__(16) unsigned char tile_smem[];
    R* const s_psi = reinterpret_cast<R*>(tile_smem);                       // [N2]
    R2* const s_u = reinterpret_cast<R2*>(s_psi + ((N2 + 1) & ~1));         // [N1]
    R* const s_ic = reinterpret_cast<R*>(s_u + N1);                         // [N1]
    R* const s_g = s_ic + N1;                                               // [4][N1] g_1 .. g_4
    __shared__ long long s_mass[16];
    __shared__ int s_abort;

    const int t = threadIdx.x, NT = blockDim.x;
    const int nx = I.nx, ny = I.ny, pitch = I.pitch;
    const unsigned plane = (unsigned)ny * (unsigned)pitch;
    const bool perx = I.flow[EW] == PERIODIC, pery = I.flow[ES] == PERIODIC;
    const bool tperx = I.therm[EW] == T_PERIODIC, tpery = I.therm[ES] == T_PERIODIC;
    const bool wallS = I.flow[ES] == WALL, wallN = I.flow[EN] == WALL;
    const R rho_ref = (R)I.rho_ref, T_ref = (R)I.T_ref, cot = (R)I.cot_theta;
    const bool use_mass = P.gravity != R(0);
    const long long step0 = __ldcg(&I.ctl->step);
    int steps = L.steps;
    if (L.targets) {
        const long long tg = __ldcg(&I.ctl->target);
        if (tg > 0) steps = (int)min((long long)steps, max(0LL, tg - step0));
    }
    if (steps == 0) return;   // the same for every CTA

    // this thread's nodes of the current tile: the one it owns and its node
    // around the tile (kind 0: outside the domain, 1: inside, 2: ghost layer of
    // a wall; the first ring, tile + 1, comes before the second).  Set up once
    // unless the CTA has several tiles.
    const int lx = t % TX, ly = t / TX;
    const int kr = t >= L.ring0 ? t - L.ring0 : t - L.ring0 + NT;
    const int c2 = (ly + 2) * W2 + lx + 2, c1 = (ly + 1) * W1 + lx + 1;
    int x0 = 0, y0 = 0, tw = 0, th = 0, n_ring1 = 0, n_ring = 0, set_up = -1;
    int gx = 0, gy = 0, oo = 0, rk = 0, rx = 0, ry = 0, ro = 0;
    bool own = false;
    auto ring_node = [&](int k, int* px, int* py, int* off) -> int {
        if (k >= n_ring) return 0;
        int d = 1;
        if (k >= n_ring1) { k -= n_ring1; d = 2; }
        const int w = tw + 2 * d, h = th + 2 * (d - 1);
        if (k < w) { *px = k - d; *py = -d; }
        else if (k < 2 * w) { *px = k - w - d; *py = th + d - 1; }
        else if (k < 2 * w + h) { *px = -d; *py = k - 2 * w - (d - 1); }
        else { *px = tw + d - 1; *py = k - 2 * w - h - (d - 1); }
        int x = x0 + *px, y = y0 + *py;
        if (perx) x = wrapi(x, nx);
        if (pery) y = wrapi(y, ny);
        if (x < 0 || x >= nx) return 0;
        if (y < 0 || y >= ny) {
            *off = x;
            return (y == -1 && wallS) || (y == ny && wallN) ? 2 : 0;
        }
        *off = y * pitch + x;
        return 1;
    };

    int err = 0;
    if (t == 0) s_abort = 0;

    for (int s = 0; s < steps; ++s) {
        const long long step = step0 + s;
        const int par = (int)(step & 1);
        const bool first = step == 0;
        const TF* const fsrc = (const TF*)I.f[par];
        const TG* const gsrc = (const TG*)I.g[par];
        const R* const Psrc = (const R*)I.P[par];
        TF* const fdst = (TF*)I.f[par ^ 1];
        TG* const gdst = (TG*)I.g[par ^ 1];
        R* const Pdst = (R*)I.P[par ^ 1];
        // the density sum of the previous step: published by the previous
        // launch, or the fixed-point sum the last step's CTAs added
        R rho_ave = R(0);
        if (use_mass) {
            const int sl = (int)((step + 2) % 3);
            const double m = s == 0 ? __ldcg(&I.ctl->mass[sl]) : mass_total(I.ctl, sl, P.m_unit);
            rho_ave = (R)(m * I.inv_n);
        }
        // this step's sum: with buoyancy every step's is read by the next;
        // without, only the last one of the launch is kept
        const bool sum_mass = use_mass || s == steps - 1;
        long long msum = 0;
        if (blockIdx.x == 0 && t == 0) {
            I.ctl->massq[(step + 1) % 3] = 0;
            I.ctl->massh[(step + 1) % 3] = 0;
        }

        for (int tile = blockIdx.x; tile < L.n_tiles; tile += gridDim.x) {
            if (tile != set_up) {
                set_up = tile;
                x0 = (tile % L.ntx) * TX;
                y0 = (tile / L.ntx) * TY;
                // the last tiles of a row or column end with the domain
                tw = min(TX, nx - x0);
                th = min(TY, ny - y0);
                n_ring1 = 2 * (tw + th) + 4;
                n_ring = n_ring1 + 2 * (tw + th) + 12;
                gx = x0 + lx;
                gy = y0 + ly;
                own = lx < tw && ly < th;
                oo = own ? gy * pitch + gx : 0;
                rk = ring_node(kr, &rx, &ry, &ro);
            }
            R fo[9], go[5], fr[9], gr[5], Pp = R(0), gpsi = R(0);
            auto load = [&](int off, R* f, R* g) {
#pragma unroll
                for (int q = 0; q < 9; ++q) f[q] = (R)ld_l2(fsrc + off + q * plane);
#pragma unroll
                for (int q = 0; q < 5; ++q) g[q] = (R)ld_l2(gsrc + off + q * plane);
            };
            if (own) {
                load(oo, fo, go);
                Pp = ld_l2(Psrc + oo);
            }
            if (rk == 1) load(ro, fr, gr);

            // psi of the ghost layer of a wall, from the populations of layers 1
            // and 2 at column x (Section 3.3)
            auto ghost = [&](int x, bool south) -> R {
                const int y1 = south ? 0 : ny - 1, y2 = south ? 1 : ny - 2;
                const int xp = perx ? wrapi(x + 1, nx) : min(x + 1, nx - 1);
                const int xm = perx ? wrapi(x - 1, nx) : max(x - 1, 0);
                auto rho_at = [&](int xx, int yy) {
                    R f[9];
#pragma unroll
                    for (int q = 0; q < 9; ++q) f[q] = (R)ld_l2(fsrc + yy * pitch + xx + q * plane);
                    return radd(sum9(f), rho_ref);
                };
                R g[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) g[q] = (R)ld_l2(gsrc + y1 * pitch + x + q * plane);
                return ghost_psi(P, rho_at(x, y2), rho_at(xp, y1), rho_at(xm, y1), cot,
                                 radd(sum5(g), T_ref), &err);
            };
            if (rk == 2) gpsi = ghost(ro, ry < 0);
            // the previous tile's stage C has read s_u, s_g and s_ic
            __syncthreads();

            // ---- A: the owned node
            Node<R> no, nr;
            auto keep = [&](const Node<R>& n, const R* g, int i2, int i1, bool near) {
                if (!(n.q2 >= R(0))) err |= (n.q2 != n.q2) ? ERR_NONFINITE : ERR_PSI;
                s_psi[i2] = n.psi;
                if (near) {
                    s_ic[i1] = blend_iC(n.C, n.iC);
#pragma unroll
                    for (int q = 0; q < 4; ++q) s_g[q * N1 + i1] = g[q + 1];
                }
            };
            if (own) {
                node_fields(P, rho_ref, T_ref, fo, go, no);
                keep(no, go, c2, c1, true);
                if (sum_mass) msum += mass_fix(P, no.rho, gy >= I.own_y0 && gy < I.own_y1);
            }
            // ---- A: the nodes around the tile
            const bool near = kr < n_ring1;
            const int r2 = (ry + 2) * W2 + rx + 2, r1 = near ? (ry + 1) * W1 + rx + 1 : 0;
            if (rk == 1) {
                node_fields(P, rho_ref, T_ref, fr, gr, nr);
                keep(nr, gr, r2, r1, near);
            } else if (rk == 2) {
                s_psi[r2] = gpsi;
            }
            for (int k = kr + NT; k < n_ring; k += NT) {
                int kx = 0, ky = 0, ko = 0;
                const int kk = ring_node(k, &kx, &ky, &ko);
                const int i2 = (ky + 2) * W2 + kx + 2;
                if (kk == 1) {
                    R f[9], g[5];
                    Node<R> n;
                    load(ko, f, g);
                    node_fields(P, rho_ref, T_ref, f, g, n);
                    const bool nk = k < n_ring1;
                    keep(n, g, i2, nk ? (ky + 1) * W1 + kx + 1 : 0, nk);
                } else if (kk == 2) {
                    s_psi[i2] = ghost(ko, ky < 0);
                }
            }
            __syncthreads();

            // ---- B: force and velocity.  Beyond an open edge the fields are
            // those of the edge node (x first, then y); beyond a wall psi is the
            // ghost layer's
            auto force = [&](const Node<R>& n, int i2, int i1, int x, int y, R2* s12, R2* F) -> R2 {
                const int dw = (!perx && x == 0) ? 0 : -1, de = (!perx && x == nx - 1) ? 0 : 1;
                const int ds = (I.flow[ES] == OPEN && y == 0) ? 0 : -W2;
                const int dn = (I.flow[EN] == OPEN && y == ny - 1) ? 0 : W2;
                const R* p = s_psi + i2;
                *s12 = force_stencil<R>(p[dw], p[de], p[ds + dw], p[ds], p[ds + de], p[dn + dw], p[dn],
                                        p[dn + de]);
                *F = force_of<R>(P, *s12, n.psi, n.rho, rho_ave);
                R2 u = pr(R(0), R(0));
                if (!P.frozen_flow) u = velocity<R>(*F, pr(n.jx, n.jy), n.ir);
                s_u[i1] = u;
                return u;
            };
            if (rk == 1 && near) {
                R2 s12, F;
                const int y = pery ? wrapi(y0 + ry, ny) : y0 + ry, x = perx ? wrapi(x0 + rx, nx) : x0 + rx;
                force(nr, r2, r1, x, y, &s12, &F);
            }
            const bool eW = gx == 0, eE = gx == nx - 1, eS = gy == 0, eN = gy == ny - 1;
            // element offsets to the neighbour columns / rows (wrapped)
            const int oW = eW ? nx - 1 : -1, oE = eE ? 1 - nx : 1;
            const int oS = eS ? (ny - 1) * pitch : -pitch, oN = eN ? (1 - ny) * pitch : pitch;
            R2 u = pr(R(0), R(0));
            if (own) {
                R2 s12, F;
                u = force(no, c2, c1, gx, gy, &s12, &F);
                TF* const fw = fdst + oo;
                if (P.frozen_flow) {
#pragma unroll
                    for (int q = 0; q < 9; ++q) st_st(fw + q * plane, (TF)fo[q]);
                } else {
                    R fs[9];
                    if constexpr (UNIT)
                        collide9_unit(P, no.rhod, pr(no.jx, no.jy), no.m7, no.m8, u, F, s12, fs, 1);
                    else
                        collide9(P, no.rho, no.rhod, fo, u, F, s12, fs, 1);
                    st_st(fw, (TF)fs[0]);
                    if (!((eW | eE) & !perx) && !((eS | eN) & !pery)) {
                        // every destination exists (periodic edges wrap)
                        st_st(fw + 1 * plane + oE, (TF)fs[1]);
                        st_st(fw + 2 * plane + oN, (TF)fs[2]);
                        st_st(fw + 3 * plane + oW, (TF)fs[3]);
                        st_st(fw + 4 * plane + oS, (TF)fs[4]);
                        st_st(fw + 5 * plane + oE + oN, (TF)fs[5]);
                        st_st(fw + 6 * plane + oW + oN, (TF)fs[6]);
                        st_st(fw + 7 * plane + oW + oS, (TF)fs[7]);
                        st_st(fw + 8 * plane + oE + oS, (TF)fs[8]);
                    } else {
                        // direction (cx, cy) of this node goes to the columns whose
                        // source it is: the next one, and at an open edge the node's
                        // own (its source beyond the edge clamps to it); likewise the
                        // rows; through a wall it returns as the opposite direction
                        const bool hasW = perx || !eW, hasE = perx || !eE;
                        const bool hasS = pery || !eS, hasN = pery || !eN;
                        auto push = [&](int i, int opp, int cx, int cy) {
                            const R v = fs[i];
                            TF* const pl = fw + i * plane;
                            const bool out_y = cy > 0 ? !hasN : (cy < 0 ? !hasS : false);
                            if (out_y && (cy > 0 ? wallN : wallS)) {
                                st_st(fw + opp * plane, (TF)v);
                                return;
                            }
                            const bool x_next = cx == 0 || (cx > 0 ? hasE : hasW);
                            const int x_off = cx == 0 ? 0 : (cx > 0 ? oE : oW);
                            const bool x_own = cx != 0 && !perx && (cx > 0 ? eW : eE);
                            const bool y_next = cy == 0 || !out_y;
                            const int y_off = cy == 0 ? 0 : (cy > 0 ? oN : oS);
                            const bool y_own = cy > 0 ? (eS && I.flow[ES] == OPEN)
                                                      : (cy < 0 && eN && I.flow[EN] == OPEN);
                            if (x_next && y_next) st_st(pl + x_off + y_off, (TF)v);
                            if (x_own && y_next) st_st(pl + y_off, (TF)v);
                            if (x_next && y_own) st_st(pl + x_off, (TF)v);
                            if (x_own && y_own) st_st(pl, (TF)v);
                        };
                        push(1, 3, 1, 0);
                        push(2, 4, 0, 1);
                        push(3, 1, -1, 0);
                        push(4, 2, 0, -1);
                        push(5, 7, 1, 1);
                        push(6, 8, -1, 1);
                        push(7, 5, -1, -1);
                        push(8, 6, 1, -1);
                    }
                }
            }
            __syncthreads();

            // ---- C: thermal stage and the blend into the destinations
            if (own) {
                const int dw = (!perx && eW) ? 0 : -1, de = (!perx && eE) ? 0 : 1;
                const bool vd = pery || !eS, vu = pery || !eN;
                const R2* const p = s_u + c1;
                const R2 z = pr(R(0), R(0));
                R2 uS0, uS1, uS2, uN0, uN1, uN2;
                if (vd || !wallS) {
                    const int d = vd ? -W1 : 0;
                    uS0 = p[d + dw]; uS1 = p[d]; uS2 = p[d + de];
                } else {
                    uS0 = uS1 = uS2 = z;
                }
                if (vu || !wallN) {
                    const int d = vu ? W1 : 0;
                    uN0 = p[d + dw]; uN1 = p[d]; uN2 = p[d + de];
                } else {
                    uN0 = uN1 = uN2 = z;
                }
                const R div12 = div12_of<R>(p[dw], p[de], uS0, uS1, uS2, uN0, uN1, uN2);
                R gs[5];
                Pdst[oo] = thermal5<UNIT>(P, go, no.Td, no.C, no.E, u, div12, Pp, first, gs);
                TG* const gw = gdst + oo;
                if (P.frozen_thermal) {
#pragma unroll
                    for (int q = 0; q < 5; ++q) st_st(gw + q * plane, go[q]);
                } else {
                    const R ic = blend_iC(no.C, no.iC);
                    st_st(gw, blend(go[0], gs[0], ic));
                    // g*_i lands on the next node as g_i + (g*_i - g_i)/(rho c_v) with
                    // that node's g_i and rho c_v; through a thermal edge it returns
                    // here as the opposite direction (halfway anti-bounce-back to
                    // the edge temperature, or bounce-back)
                    auto move = [&](int i, int opp, bool out, int off, int l, int edge) {
                        if (!out) {
                            st_st(gw + i * plane + off, blend(s_g[(i - 1) * N1 + c1 + l], gs[i], s_ic[c1 + l]));
                        } else {
                            R A = gs[i];
                            if (I.therm[edge] == T_DIRICHLET) {
                                const R tw = (R)((edge == ES ? wall_T(I, ES, gx) : I.T_edge[edge]) - I.T_ref);
                                A = rsub(rmul(rmul(R(2), P.w5_1), tw), A);
                            }
                            st_st(gw + opp * plane, blend(go[opp], A, ic));
                        }
                    };
                    move(1, 3, !tperx && eE, oE, 1, EE);
                    move(2, 4, !tpery && eN, oN, W1, EN);
                    move(3, 1, !tperx && eW, oW, -1, EW);
                    move(4, 2, !tpery && eS, oS, -W1, ES);
                }
            }
        }

        // ---- the step's density sum (exact, order-free)
        if (sum_mass) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(0xffffffffu, msum, o);
            if ((t & 31) == 0) s_mass[t >> 5] = msum;
        }
        __syncthreads();
        if (t == 0) {
            if (sum_mass) {
                long long m = 0;
                for (int w = 0; w < (NT + 31) / 32; ++w) m += s_mass[w];
                mass_add(I.ctl, (int)(step % 3), m);
            }
            __threadfence();
            const unsigned done = bar_add(L.bar);
            const unsigned all = (unsigned)(s + 1) * gridDim.x;
            if (done >= BAR_LEFT) {
                s_abort = 1;
            } else if (s == steps - 1) {
                // the last CTA of the launch publishes the density sum, advances
                // the step counter and clears the grid counter for the next launch
                if (done == all - 1) {
                    I.ctl->mass[step % 3] = mass_total(I.ctl, (int)(step % 3), P.m_unit);
                    I.ctl->step = step + 1;
                    *L.bar = 0u;
                    __threadfence();
                }
            } else if (done != all - 1) {
                const unsigned c0 = (unsigned)clock();
                unsigned v;
                while ((v = bar_load(L.bar)) < all) {
                    if ((unsigned)clock() - c0 > L.wait) {
                        atomicOr(L.bar, BAR_LEFT);
                        err |= ERR_TIMEOUT;
                        s_abort = 1;
                        break;
                    }
                }
                if (v >= BAR_LEFT) s_abort = 1;
            }
        }
        __syncthreads();
        if (s_abort) break;
    }
    if (err) atomicOr(&I.ctl->err, err);
}

// CTAs per SM of both instantiations, the fewer: a plan outlives lbm_reconfigure,
// which may change between unit and general rates
template <int PREC>
int tile_occ(int threads, size_t smem, int* ctas) {
    int unit = 0, general = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&unit, k_tile<PREC, true>, threads, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&general, k_tile<PREC, false>, threads, smem) !=
            cudaSuccess)
        return -1;
    *ctas = std::min(unit, general);
    return 0;
}

template <int PREC, bool UNIT>
cudaError_t tile_run(const TileLaunch& L, const PhysD& phys, int grid, int threads, size_t smem,
                     cudaStream_t st) {
    Phys<typename Types<PREC>::R> P = make_phys<typename Types<PREC>::R>(phys);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = L.steps > 1 ? 1 : 0;   // one step has no barrier
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_tile<PREC, UNIT>, L, P);
    if (e != cudaSuccess) cudaGetLastError();   // the caller answers it
    return e;
}

template <int PREC>
cudaError_t tile_run_any(const TileLaunch& L, const PhysD& phys, int grid, int threads, size_t smem,
                         cudaStream_t st) {
    return unit_rates(phys) ? tile_run<PREC, true>(L, phys, grid, threads, smem, st)
                            : tile_run<PREC, false>(L, phys, grid, threads, smem, st);
}

}  // namespace

// Which tile, and whether the domain takes this form at all.
//
// FP32 / FP16-g: a step is bound by latency (grid barrier 1.3-1.7 us, loads, three
// barriers of the CTA per tile): about 1.6 us and, per round of resident tiles,
// 3.45 us for 32 x 8 nodes (two CTAs per SM), 2.4 for 32 x 10 and 2.75 for 32 x
// 12 (one).  Which one wastes least of its last round decides (us per step, 32
// x 8 / 32 x 10 / 32 x 12): 256^2 5.1 / 7.3 / 7.6, 400 x 200 FP16-g 8.8 / 7.7 / 7.9,
// 300 x 600 pool 12.6 / 12.9 / 13.7, 512^2 15.2 / 16.8 / 15.0, 700^2 22.7 / 28.3 / 25.1.
// Over 60 sizes from 64 to 768 (136 runs, open domains and pools) the choice is 2 %
// off the best of the four on average, 16 % at most (358 x 713, open).
// Full rows of 128 bytes beat 16 x 16, 16 x 8 and 8 x 8 everywhere except where 8
// x 8 tiles with their surrounding nodes on threads of their own (one pass of
// stage A instead of two) leave at most one per SM: 64^2 4.0 -> 3.35 us.  Against
// the sweep with its best tile, 512^2 is 15.1 us against 23.5, 768^2 28.7 (8
// rounds of 32 x 8) against 28.7 and 1024^2 48.5 against 40.6: up to 26 us here.
// Walls, a heater and buoyancy add up to 2.5 us that this does not model, and cost
// the sweep as much: pools at the limit, 700^2 24.6 against 27.5 us, 735^2 24.8
// against 28.0, FP16-g 735^2 26.3 against 30.4, FP64 600^2 173 against 175.
//
// FP64: each of an SM's four partitions takes 64 cycles per FP64 warp
// instruction, so the time is that of the busiest partition: about 170
// instructions per warp of owned nodes, 65 per warp of surrounding nodes (90
// in the first ring).  The candidates are compared by that count.  Measured /
// modelled us per step: 64^2 8 x 4 with separate surrounding threads 8.3 / 8.7
// (16 x 8 12.1 / 11.4), 200^2 20 x 14 21.5 / 23.3 (32 x 8 35.7 / 37.3), 384^2
// 32 x 8 71.1 / 74.6; the sweep needs 87 at 200^2, 149 at 384^2, 165 at 500^2
// (this form 122) and 209 at 610^2, where 205 are modelled for 11 rounds of 32 x 8,
// so domains up to 190 modelled microseconds come here.
int tile_plan(int prec, const Inst& I, int sms, int want_tx, int want_ty, TilePlan* out) {
    out->tx = 0;
    const bool any = want_tx > 0;
    if ((long long)I.nx * I.ny > (1 << 20)) return 0;   // far beyond either limit below
    struct Cand { int tx, ty, sep; };
    static const Cand c32[4] = {{8, 8, 1}, {32, 8, 0}, {32, 10, 0}, {32, 12, 0}};
    static const Cand c64[5] = {{8, 4, 1}, {8, 8, 1}, {32, 8, 0}, {16, 8, 0}, {20, 14, 0}};
    const Cand* const cand = prec == 0 ? c64 : c32;
    const int n_cand = prec == 0 ? 5 : 4;
    const size_t es = prec == 0 ? 8 : 4;
    double best = 1e30;
    for (int k = 0; k < n_cand; ++k) {
        const int tx = cand[k].tx, ty = cand[k].ty;
        if (any && (tx != want_tx || ty != want_ty)) continue;
        const int n_ring1 = 2 * (tx + ty) + 4, n_ring = n_ring1 + 2 * (tx + ty) + 12;
        const int own_w = (tx * ty + 31) / 32, ring_w = (n_ring + 31) / 32;
        // separate: the surrounding nodes have threads of their own
        const int ring0 = cand[k].sep ? own_w * 32 : 0;
        const int threads = cand[k].sep ? (own_w + ring_w) * 32 : std::max(own_w * 32, (n_ring1 + 31) / 32 * 32);
        const long long ntx = (I.nx + tx - 1) / tx, nt = ntx * ((I.ny + ty - 1) / ty);
        const size_t smem = tile_bytes(es, tx, ty);
        int ctas = 0;
        const int rc = prec == 0 ? tile_occ<0>(threads, smem, &ctas)
                       : prec == 1 ? tile_occ<1>(threads, smem, &ctas)
                                   : tile_occ<2>(threads, smem, &ctas);
        if (rc) return -1;
        if (ctas < 1) continue;
        const long long slots = (long long)ctas * sms, rounds = (nt + slots - 1) / slots;
        double us;
        if (prec != 0) {
            if (cand[k].sep && nt > sms && !any) continue;
            static const double per_round[4] = {1.75, 3.45, 2.4, 2.75};
            us = 1.6 + per_round[k] * (double)rounds;
            if (us > 26.0 && !any) continue;
        } else {
            const double ring_cost = 65.0 + 25.0 * n_ring1 / n_ring;
            // the busiest partition of one CTA, and all partitions of the CTAs
            // that share an SM
            const double part = (own_w + 3) / 4 * 170.0 +
                                (cand[k].sep ? 0.0 : (ring_w + 3) / 4 * ring_cost);
            const long long share = std::min<long long>(ctas, (nt + sms - 1) / sms);
            const double all = (double)share * (own_w * 170.0 + ring_w * ring_cost) / 4.0;
            us = (double)rounds * (3.4 + std::max(part, all) * 64.0 / 2070.0);
            if (tx * ty == 128) us *= 1.12;   // measured against modelled, 64^2 and 384^2
            if (us > 190.0 && !any) continue;
        }
        if (us >= best) continue;
        best = us;
        out->tx = tx;
        out->ty = ty;
        out->ring0 = ring0;
        out->threads = threads;
        out->ntx = (int)ntx;
        out->n_tiles = (int)nt;
        out->grid = (int)((nt + rounds - 1) / rounds);
        out->smem = smem;
    }
    return 0;
}

cudaError_t tile_launch(int prec, const TilePlan& T, const TileLaunch& L, const PhysD& phys,
                        cudaStream_t st) {
    if (prec == 0) return tile_run_any<0>(L, phys, T.grid, T.threads, T.smem, st);
    if (prec == 1) return tile_run_any<1>(L, phys, T.grid, T.threads, T.smem, st);
    return tile_run_any<2>(L, phys, T.grid, T.threads, T.smem, st);
}

}  // namespace lbm
