// Interface analyses of the density field, on the device:
//  * the contact angle of a sessile droplet (Section 4.2 relaxes the droplet
//    without evaporation until it shows the prescribed angle, then heats);
//  * the 4-connected regions of the vapour (or liquid) phase, from which the
//    departure of a bubble from the heated wall and its size follow
//    (Section 4.3, the Fritz relation D_d ~ g^-1/2).
//
// Contact angle.  Every lattice link between horizontally or vertically
// adjacent nodes whose densities lie on opposite sides of rho_mid contributes
// one interface point, placed on the link by linear interpolation; links
// with a node below row skip_rows are left out.  Two passes over the field
// accumulate, in double, first the count and mean of the points and then the
// centred moment sums of the algebraic circle fit
//   min sum (u^2 + v^2 + D u + E v + F)^2,  (u, v) = point - mean,
// which the host solves for the circle.  Each pass keeps per-block partials
// and the last block to finish folds them in block order, so the result does
// not depend on scheduling.
//
// Regions.  A union-find over node indices: every node in the phase starts
// with the first node of its run within 32 columns as parent; runs that touch
// (across the seams of periodic axes too) have their roots merged by an atomicMin that
// makes the larger root point to the smaller one, so a parent index is never
// above its node's index and every region ends with its smallest node index
// as root.  Loops that chase parents or retry a merge strictly decrease an
// index, so they end within n iterations; they are still capped and report
// an error word instead of running on.  A flattening pass then writes each
// node's root, and a statistics pass accumulates per-root area, row sums,
// row range and edge contacts with atomics, one lane for all lanes of a warp
// that share a root (integers only: the result is exact and independent of
// order).  2048^2 with 440 bubbles: merging 254 -> 71 us, the
// other passes 103 -> 68.
#include <algorithm>

#include "lbm_internal.cuh"

namespace lbm {

namespace {

enum { ANA_BLOCKS = 304, ANA_THREADS = 256, ANA_VALS = 9 };

struct IfaceScratch {
    double partial[ANA_BLOCKS * ANA_VALS];
    double mean[ANA_VALS];
    unsigned ticket;
};

__device__ __forceinline__ void add_point(double* v, int pass, const double* mean, double px,
                                          double py) {
    if (pass == 0) {
        v[0] += 1.0;
        v[1] += px;
        v[2] += py;
    } else {
        const double u = px - mean[1] / mean[0], w = py - mean[2] / mean[0];
        const double z = u * u + w * w;
        v[0] += 1.0;
        v[1] += u;
        v[2] += w;
        v[3] += u * u;
        v[4] += w * w;
        v[5] += u * w;
        v[6] += u * z;
        v[7] += w * z;
        v[8] += z;
    }
}

__global__ void __launch_bounds__(ANA_THREADS)
    k_iface(const double* __restrict__ rho, int nx, int ny, double rho_mid, int skip, int pass,
            double* out, IfaceScratch* sc) {
    __shared__ double red[ANA_VALS][ANA_THREADS / 32];
    __shared__ bool last;
    double v[ANA_VALS] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    const double* mean = sc->mean;
    const long long n = (long long)nx * (ny - skip);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx), y = skip + (int)(i / nx);
        const long long c = (long long)y * nx + x;
        const double a = rho[c] - rho_mid;
        if (x + 1 < nx) {
            const double b = rho[c + 1] - rho_mid;
            if ((a >= 0.0) != (b >= 0.0)) add_point(v, pass, mean, x + a / (a - b), (double)y);
        }
        if (y + 1 < ny) {
            const double b = rho[c + nx] - rho_mid;
            if ((a >= 0.0) != (b >= 0.0)) add_point(v, pass, mean, (double)x, y + a / (a - b));
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = 0; k < ANA_VALS; ++k) {
        double x = v[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[k][wid] = x;
    }
    __syncthreads();
    if (threadIdx.x < ANA_VALS) {
        const int k = threadIdx.x;
        double x = red[k][0];
        for (int w = 1; w < ANA_THREADS / 32; ++w) x += red[k][w];
        sc->partial[blockIdx.x * ANA_VALS + k] = x;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) {
        // one warp per value: lane l adds blocks l, l + 32, ... in order, then
        // the lanes pairwise (a fixed order)
        __threadfence();
        for (int k = wid; k < ANA_VALS; k += ANA_THREADS / 32) {
            double x = 0.0;
            for (unsigned b = lane; b < gridDim.x; b += 32) x += __ldcg(&sc->partial[b * ANA_VALS + k]);
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (lane != 0) continue;
            if (pass == 0) sc->mean[k] = x;
            else out[k] = x;
            if (pass == 1 && k < 3) out[ANA_VALS + k] = sc->mean[k];
            if (k == 0) sc->ticket = 0u;
        }
    }
}

// ---- regions -----------------------------------------------------------
enum { CC_THREADS = 256 };

struct CCArrays {
    unsigned long long* sum_y;
    int* parent;
    unsigned* area;
    int* y_min;
    int* y_max;
    int* flags;     // bit 0 W, 1 E, 2 S, 3 N
    int* roots;
    int* count;     // [0] roots found, [1] error word
};

__device__ __forceinline__ int find_root(const int* parent, int x, long long cap, int* err) {
    long long it = 0;
    int p = __ldcg(&parent[x]);
    while (p != x) {
        x = p;
        p = __ldcg(&parent[x]);
        if (++it > cap) {
            atomicOr(err, 1);
            break;
        }
    }
    return x;
}

// Nodes are taken in segments of 32 columns of a row, one warp each: every node
// of the phase starts with the first node of its run inside the segment as
// parent (a ballot), so that only runs have to be merged and parent chains
// stay short.
struct Seg {
    int x, y, lane;
    long long i;        // node index
    bool in;            // the column exists
};
__device__ __forceinline__ Seg seg_of(long long s, int segs, int nx) {
    Seg g;
    g.lane = threadIdx.x & 31;
    g.y = (int)(s / segs);
    g.x = (int)(s % segs) * 32 + g.lane;
    g.in = g.x < nx;
    g.i = (long long)g.y * nx + g.x;
    return g;
}
// warps of the grid, and this thread's
__device__ __forceinline__ long long warp_id() { return ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ long long warp_count() { return ((long long)gridDim.x * blockDim.x) >> 5; }

__global__ void k_cc_init(const double* __restrict__ rho, int nx, int ny, double thr, int below,
                          CCArrays A) {
    const int segs = (nx + 31) / 32;
    for (long long s = warp_id(); s < (long long)segs * ny; s += warp_count()) {
        const Seg g = seg_of(s, segs, nx);
        bool in = false;
        if (g.in) {
            const double r = rho[g.i];
            in = below ? (r < thr) : (r > thr);
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (!g.in) continue;
        // the run's first lane: one past the last lane below this one that is out
        const unsigned out_below = ~m & ((1u << g.lane) - 1u);
        const int first = out_below ? 32 - __clz(out_below) : 0;
        A.parent[g.i] = in ? (int)(g.i - g.lane + first) : -1;
        A.area[g.i] = 0u;
        A.sum_y[g.i] = 0ull;
        A.y_min[g.i] = 0x7fffffff;
        A.y_max[g.i] = -1;
        A.flags[g.i] = 0;
    }
}

__device__ void unite(int* parent, int a, int b, long long cap, int* err) {
    for (long long it = 0; it <= cap; ++it) {
        a = find_root(parent, a, cap, err);
        b = find_root(parent, b, cap, err);
        if (a == b) return;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        // link the larger root b under a; if b stopped being a root meanwhile,
        // continue from its new parent
        const int old = atomicMin(&parent[b], a);
        if (old == b) return;
        b = old;
    }
    atomicOr(err, 2);
}

__global__ void k_cc_union(int nx, int ny, int perx, int pery, CCArrays A) {
    const long long n = (long long)nx * ny;
    const int segs = (nx + 31) / 32;
    for (long long s = warp_id(); s < (long long)segs * ny; s += warp_count()) {
        const Seg g = seg_of(s, segs, nx);
        const bool in = g.in && __ldcg(&A.parent[g.i]) >= 0;
        // west: a run that goes on in the segment before (or across the seam)
        if (in && g.lane == 0) {
            const int xw = g.x > 0 ? g.x - 1 : (perx ? nx - 1 : -1);
            const long long j = (long long)g.y * nx + xw;
            if (xw >= 0 && j != g.i && __ldcg(&A.parent[j]) >= 0)
                unite(A.parent, (int)g.i, (int)j, n, &A.count[1]);
        }
        // north: one merge per stretch of columns that this row's and the next
        // row's runs have in common
        const int yn = g.y + 1 < ny ? g.y + 1 : (pery ? 0 : -1);
        const long long j = (long long)yn * nx + g.x;
        const bool both = in && yn >= 0 && j != g.i && __ldcg(&A.parent[j]) >= 0;
        const unsigned m = __ballot_sync(0xffffffffu, both);
        if (both && (g.lane == 0 || !(m >> (g.lane - 1) & 1u)))
            unite(A.parent, (int)g.i, (int)j, n, &A.count[1]);
    }
}

__global__ void k_cc_flatten(long long n, CCArrays A) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        if (A.parent[i] >= 0) A.parent[i] = find_root(A.parent, (int)i, n, &A.count[1]);
}

// per-root sums: one lane per root and segment adds for the lanes that share it
__global__ void k_cc_stats(int nx, int ny, int max_roots, CCArrays A) {
    const int segs = (nx + 31) / 32;
    for (long long s = warp_id(); s < (long long)segs * ny; s += warp_count()) {
        const Seg g = seg_of(s, segs, nx);
        const int r = g.in ? A.parent[g.i] : -1;
        const unsigned same = __match_any_sync(0xffffffffu, r);
        if (r < 0) continue;
        const int f = (g.x == 0 ? 1 : 0) | (g.x == nx - 1 ? 2 : 0) | (g.y == 0 ? 4 : 0) | (g.y == ny - 1 ? 8 : 0);
        if (f & 3) atomicOr(&A.flags[r], f);
        if (g.lane == __ffs(same) - 1) {
            const unsigned k = (unsigned)__popc(same);
            atomicAdd(&A.area[r], k);
            atomicAdd(&A.sum_y[r], (unsigned long long)g.y * k);
            atomicMin(&A.y_min[r], g.y);
            atomicMax(&A.y_max[r], g.y);
            if (f & 12) atomicOr(&A.flags[r], f & 12);
        }
        if (r == (int)g.i) {
            const int slot = atomicAdd(&A.count[0], 1);
            if (slot < max_roots) A.roots[slot] = r;
        }
    }
}

__global__ void k_cc_gather(const int* roots, int m, CCArrays A, RegionOut* out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= m) return;
    const int r = roots[k];
    RegionOut o;
    o.label = r;
    o.area = A.area[r];
    o.sum_y = (long long)A.sum_y[r];
    o.y_min = A.y_min[r];
    o.y_max = A.y_max[r];
    o.flags = A.flags[r];
    out[k] = o;
}

// sum_y (8n bytes) | parent, area, y_min, y_max, flags, roots (4n each) | count
CCArrays cc_arrays(void* scratch, long long n) {
    char* p = (char*)scratch;
    CCArrays A;
    A.sum_y = (unsigned long long*)p;
    A.parent = (int*)(p + 8 * n);
    A.area = (unsigned*)(p + 12 * n);
    A.y_min = (int*)(p + 16 * n);
    A.y_max = (int*)(p + 20 * n);
    A.flags = (int*)(p + 24 * n);
    A.roots = (int*)(p + 28 * n);
    A.count = (int*)(p + 32 * n);
    return A;
}

int grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 4096) b = 4096;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

size_t iface_scratch_bytes() { return sizeof(IfaceScratch); }

int iface_launch(const double* rho, int nx, int ny, double rho_mid, int skip, double* out12,
                 void* scratch, cudaStream_t st) {
    if (skip >= ny) skip = ny;
    IfaceScratch* sc = (IfaceScratch*)scratch;
    // small fields take fewer blocks: their fold is what they would wait for
    const long long n = (long long)nx * (ny - skip);
    const int blocks = (int)std::min<long long>(ANA_BLOCKS, std::max<long long>(1, (n + 511) / 512));
    for (int pass = 0; pass < 2; ++pass)
        k_iface<<<blocks, ANA_THREADS, 0, st>>>(rho, nx, ny, rho_mid, skip, pass, out12, sc);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

size_t regions_scratch_bytes(long long n) { return (size_t)n * 32 + 64; }

int regions_launch(const double* rho, int nx, int ny, int perx, int pery, double thr, int below,
                   void* scratch, int max_roots, int** parent_out, int** roots_out,
                   int** count_out, cudaStream_t st) {
    const long long n = (long long)nx * ny;
    const CCArrays A = cc_arrays(scratch, n);
    if (cudaMemsetAsync(A.count, 0, 2 * sizeof(int), st) != cudaSuccess) return -1;
    // whole warps per segment of 32 columns
    const int g = grid_for((long long)((nx + 31) / 32 * 32) * ny, CC_THREADS);
    k_cc_init<<<g, CC_THREADS, 0, st>>>(rho, nx, ny, thr, below, A);
    k_cc_union<<<g, CC_THREADS, 0, st>>>(nx, ny, perx, pery, A);
    k_cc_flatten<<<g, CC_THREADS, 0, st>>>(n, A);
    k_cc_stats<<<g, CC_THREADS, 0, st>>>(nx, ny, max_roots < n ? max_roots : (int)n, A);
    *parent_out = A.parent;
    *roots_out = A.roots;
    *count_out = A.count;
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int regions_gather_launch(void* scratch, long long n, int m, RegionOut* out, cudaStream_t st) {
    const CCArrays A = cc_arrays(scratch, n);
    if (m <= 0) return 0;
    k_cc_gather<<<(m + 127) / 128, 128, 0, st>>>(A.roots, m, A, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace lbm
