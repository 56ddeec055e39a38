// The coarse part of the multigrid cycle in one launch: every level up to
// `top`, the highest level that covers the whole domain and fits (levels 1
// and up hold the boxes of a uniformly refined part of the tree; below level 1
// lie the grids of N/2, ..., 2 cells per root box, arXiv:1701.04329 Sec. 3.2,
// which exist only here).  A level is one rectangular grid without refinement
// boundaries, so the V-cycle below and at `top` needs from global memory only
// level top's solution and source term (and the domain face data), and gives
// back level top's solution.
//
// Why one launch: a per-level launch of a few boxes takes 2-4 us whatever it
// computes, and a V-cycle makes 11 of them per level.  Here a step costs a
// block barrier and a few shared-memory latencies.  The grids of one tree
// are spread over the R thread blocks of a cluster (R = 1: one block), in
// slabs along the last axis; a value next to a slab's edge is also stored
// into the neighbour block's halo plane (distributed shared memory), and the
// steps end with a cluster barrier.  Grids too small to be worth it are held
// whole by every block and computed by each of them alike: only the
// restriction into the first such grid crosses blocks.
//
// Shared memory of a level: u, v' and the source with a ghost layer.  The
// ghost of a domain side depends on nothing but the cell inside
// (g = 2b - u_1, u_1 + h b, or the cell at the other end of a periodic row),
// so whoever stores that cell stores the ghost too, and the steps read their
// neighbours without a branch; the ghost slots of the source hold b.  v' of
// level top stays in global memory.
//
// Variable coefficients (VAR; kernels_var_staged.cuh): every level's 2D + 2
// coefficient arrays lie in shared memory too, copied from a packed image that
// is gathered once per eps (mode 3).
//
// What bounds a step is its own chain of instructions: it runs once per warp,
// so its instruction fetches count as much as its shared-memory latencies.
// The steps are therefore short: one copy for all levels (the sizes are
// run-time values), no unrolled batches, 32-bit shared-memory addressing, and
// an all-Dirichlet instance (BC = false) without the other sides' rules.
//
// Measured on a GB300 at 2 GHz, one V-cycle's visit: 2D, 64^2 and below, FP64
// 63 us (levels 3-4 as 22 launches and a one-block bottom up to 32^2 before:
// 120 us), FP32 30 us (77 us); 3D on eight blocks, FP64, 16^3 and below, 62 us
// (11 launches and a one-block bottom before: 87 us), FP32 up to 32^3 for one
// tree, 50 us with cold caches (16^3 and below alone 28 us, 49 us before).
// Whole solves: 31 k unknowns in 2D, FP64, 2.89 -> 2.22 ms; 73 k unknowns on
// a 3 x 2 block of root boxes, mixed, 7.40 -> 4.67 ms; 12 small quadtrees,
// FP64, 2.30 -> 1.82 ms.  With variable coefficients (every level below them
// on per-level launches before): 107 k unknowns in 2D, FP64, 6.57 -> 3.56 ms;
// (r,z), 294 k, mixed, 5.80 -> 2.50 ms; 3D, 3.5 M, mixed, 7.96 -> 5.70 ms.  A
// half-sweep of a small grid is then 225 cycles in FP32; in FP64 about 1100, of
// which the exact neighbour sum takes 285 and every dependent FP64 operation
// 64-76.  A cluster barrier costs 350-450.
#pragma once
#include "coarse_plan.h"
#include "kernels.cuh"
#include "kernels_smooth.cuh"  // cp_async
#include "var_ops.cuh"

namespace afg {

extern __shared__ __align__(16) unsigned char co_smem[];
constexpr int kCoarseHead = (sizeof(CoarseArgs) + 15) / 16 * 16;  // the plan, ahead of the grids

__device__ __forceinline__ const CoarseArgs &co_plan() { return *reinterpret_cast<const CoarseArgs *>(co_smem); }
template <typename T>
__device__ __forceinline__ T *co_mem() { return reinterpret_cast<T *>(co_smem + kCoarseHead); }

__device__ __forceinline__ unsigned co_map(const void *p, int rank) {  // address of p in block `rank` of the cluster
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void co_store(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void co_store(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// every thread of every block of the cluster; orders shared-memory stores, remote ones included
__device__ __forceinline__ void co_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void co_sync(int nr) {
    if (nr > 1) co_cluster_sync();
    else __syncthreads();
}

// 2^e, exactly (an FP64 division takes about a thousand cycles of a lone warp)
template <typename T>
__device__ __forceinline__ T co_pow2(int e) {
    if constexpr (sizeof(T) == 8) return __longlong_as_double((long long)(1023 + e) << 52);
    else return __int_as_float((127 + e) << 23);
}

// one level's slab of this block; u, v, r: first element of the level's arrays
template <int D, typename T>
struct CoLevel {
    int nx, ny, P, nr, z0;  // cells per row, rows per plane (1 in 2D), planes of this slab, slabs, first plane
    int W, PS;              // padded row, padded plane
    int u, v, r;
    int lg;                 // cell size 2^-lg (unit root boxes)
    __device__ __forceinline__ T h() const { return co_pow2<T>(-lg); }
    __device__ __forceinline__ CoLevel(int li, int rank) {
        const CoarseArgs &S = co_plan();
        nx = S.nx[li];
        ny = D == 3 ? S.ny[li] : 1;
        P = S.P[li];
        nr = S.nr[li];
        z0 = nr > 1 ? rank * P : 0;
        W = nx + 2;
        PS = D == 3 ? W * (ny + 2) : W;
        u = S.ou[li];
        v = S.ov[li];
        r = S.orh[li];
        lg = li + 1;
    }
    __device__ __forceinline__ int slot(int i, int j, int k) const {
        return (k + 1) * PS + (D == 3 ? (j + 1) * W : 0) + i + 1;
    }
};

// c / d by a multiplication, magic = ceil(2^32 / d) (0 for d = 1); exact for c d < 2^32
__device__ __forceinline__ int co_div(int c, unsigned magic) { return magic ? (int)__umulhi((unsigned)c, magic) : c; }

// entry c of rows of w entries -> position in the row, row, plane (local)
template <int D>
__device__ __forceinline__ void co_decode(int c, int w, unsigned mw, int ny, unsigned my, int &x, int &j, int &k) {
    const int row = co_div(c, mw);
    x = c - row * w;
    if (D == 3) {
        k = co_div(row, my);
        j = row - k * ny;
    } else {
        k = row;
        j = 0;
    }
}

// The planes next to a slab: addresses of the array in the blocks that hold
// them, 0 where the domain ends (periodic: the block at the other end, which
// may be this one)
struct CoEdge {
    unsigned lo, hi;
};
template <typename T>
__device__ __forceinline__ CoEdge co_edge(int nr, int rank, int array, bool periodic) {
    const int n = nr > 1 ? nr : 1, me = nr > 1 ? rank : 0;
    int lo = me > 0 ? me - 1 : (periodic ? n - 1 : -1);
    int hi = me < n - 1 ? me + 1 : (periodic ? 0 : -1);
    if (nr == 1 && lo >= 0) lo = hi = rank;
    const T *a = co_mem<T>() + array;
    CoEdge E;
    E.lo = lo < 0 ? 0u : co_map(a, lo);
    E.hi = hi < 0 ? 0u : co_map(a, hi);
    return E;
}

// ghost of a side next to a stored value (b: its boundary value; not HB: 0)
template <typename T, bool BC, bool HB>
__device__ __forceinline__ T co_ghost(T b, bool neumann, T h, T val) {
    if (BC && neumann) return HB ? fma(h, b, val) : val;
    return HB ? fma(T(2), b, -val) : -val;
}

// Stores cell (i, j, k) of array a (slot p) and every ghost that depends on
// it (one per axis at most: a level has two cells or more along every axis).
// HB: the ghosts take the boundary data; otherwise they are homogeneous.
// bc = Neumann sides | periodic axes << 6.
template <int D, typename T, bool BC, bool HB>
__device__ __forceinline__ void co_put(const CoLevel<D, T> &L, int a, const CoEdge &E, int bc, int p, int i, int j,
                                       int k, T val) {
    T *sm = co_mem<T>();
    T *A = sm + a + p;
    const T *B = sm + L.r + p;
    const int ox = i == 0 ? -1 : (i == L.nx - 1 ? 1 : 0);
    const int oy = D == 3 ? (j == 0 ? -1 : (j == L.ny - 1 ? 1 : 0)) : 0;
    const int oz = k == 0 ? -1 : (k == L.P - 1 ? 1 : 0);
    T bx = T(0), by = T(0), bz = T(0);
    if (HB) {  // read together, whether at a side or not
        bx = B[ox];
        if (D == 3) by = B[oy * L.W];
        bz = B[oz * L.PS];
    }
    A[0] = val;
    if (ox) {
        if (BC && (bc & 64)) A[-ox * L.nx] = val;
        else A[ox] = co_ghost<T, BC, HB>(bx, (bc >> (ox > 0)) & 1, L.h(), val);
    }
    if (D == 3 && oy) {
        if (BC && (bc & 128)) A[-oy * L.ny * L.W] = val;
        else A[oy * L.W] = co_ghost<T, BC, HB>(by, (bc >> (2 + (oy > 0))) & 1, L.h(), val);
    }
    if (oz) {
        const unsigned e = oz < 0 ? E.lo : E.hi;
        if (e) co_store(e + (unsigned)sizeof(T) * (p - oz * L.P * L.PS), val);
        else A[oz * L.PS] = co_ghost<T, BC, HB>(bz, (bc >> (2 * (D - 1) + (oz > 0))) & 1, L.h(), val);
    }
}

// One cell of a thread that relaxes the same cells in every half-sweep: its
// slot, scaled source, and per axis the ghost that depends on it (offset of
// its slot, 0 for none; value fma(m, b, +-u)).
template <int D, typename T, bool VAR>
struct CoCell {
    int p, ox, oy, oz;
    T c[VAR ? 2 * D + 2 : 1];  // VAR: the coefficient arrays' values
    T rs, mx, bx, my, by, mz, bz;
    bool nx, ny, nz;  // the ghost takes +u (Neumann, periodic), not -u
};

template <typename T, bool BC, bool HB>
__device__ __forceinline__ T co_ghost_of(T m, T b, bool plus, T val) {
    const T v = BC && plus ? val : -val;
    return HB ? fma(m, b, v) : v;
}

// the neighbours of a cell in the order -x, +x, -y, +y, -z, +z
template <int D, typename T>
__device__ __forceinline__ void co_neighbours(const T *a, int W, int PS, T (&x)[2 * D]) {
    x[0] = a[-1];
    x[1] = a[1];
    if constexpr (D == 3) {
        x[2] = a[-W];
        x[3] = a[W];
    }
    x[2 * D - 2] = a[-PS];
    x[2 * D - 1] = a[PS];
}

// sum_s c_s u_s of the cell at a, its coefficients at c, n apart
template <int D, typename T>
__device__ __forceinline__ T co_dot(const T *c, int n, const T *a, int W, int PS) {
    T x[2 * D], k[2 * D];
    co_neighbours<D, T>(a, W, PS, x);
#pragma unroll
    for (int s = 0; s < 2 * D; ++s) k[s] = c[s * n];
    return var_dot<D, T>(k, x);
}

// Red-black steps, one barrier per half-sweep (cells of one colour read only
// the other): u = sum/(2D) - h^2 rho/(2D).  A thread keeps its place (h, j)
// in the planes and walks along the last axis.  Where that leaves it one cell
// of each colour at most, everything about them but u stays in registers, and
// a half-sweep is the loads of the neighbours, the sum and the stores.
template <int D, typename T, bool BC, bool HB, bool VAR>
__device__ __noinline__ void co_smooth(int li, int steps, int rank, int bc) {
    const CoarseArgs &S = co_plan();
    T *sm = co_mem<T>();
    const CoLevel<D, T> L(li, rank);
    const CoEdge E = co_edge<T>(L.nr, rank, L.u, BC && ((bc >> (6 + D - 1)) & 1));
    const int hx = L.nx >> 1, plane = hx * L.ny, ng = S.ng[li], nt = blockDim.x;
    const int g = ng > 1 ? co_div(threadIdx.x, S.mp[li]) : 0;
    const int first = threadIdx.x - g * plane;
    const T inv = T(1) / T(2 * D), chat = (T(-1) / T(2 * D)) * co_pow2<T>(-2 * L.lg);
    const T h2 = co_pow2<T>(-2 * L.lg);
    const T *cf = sm + S.oc[li];
    T *u = sm + L.u;
    const T *r = sm + L.r;
    const unsigned mh = S.mh[li];
    if (L.P <= ng && plane <= nt) {
        const bool on = g < L.P && first < plane;
        CoCell<D, T, VAR> c[2];
        unsigned far = 0;  // address of the array in the block across the slab's edge
        if (on) {
            const int j = D == 3 ? co_div(first, mh) : 0, x = first - j * hx, par = (j + L.z0 + g + D) & 1;
            const int oy = D == 3 ? (j == 0 ? -1 : (j == L.ny - 1 ? 1 : 0)) : 0;
            const int oz = g == 0 ? -1 : (g == L.P - 1 ? 1 : 0);
            if (oz) far = oz < 0 ? E.lo : E.hi;
#pragma unroll
            for (int q = 0; q < 2; ++q) {  // q: colour
                CoCell<D, T, VAR> &w = c[q];
                const int up = q ? 1 - par : par;  // the cell at i = 2x + up
                const int ox = up ? (x == hx - 1 ? 1 : 0) : (x == 0 ? -1 : 0);
                w.p = L.slot(2 * x + up, j, g);
                w.rs = r[w.p] * (VAR ? -h2 : chat);  // -h^2 rho, exactly, or -h^2 rho / (2D)
                if (VAR) {
#pragma unroll
                    for (int f = 0; f < 2 * D + 2; ++f) w.c[f] = cf[f * S.csz[li] + w.p];
                }
                auto side = [&](int axis, int o, int stride, int n, int &off, T &m, T &b, bool &plus) {
                    const int s = 2 * axis + (o > 0);
                    const bool per = BC && ((bc >> (6 + axis)) & 1), neu = BC && ((bc >> s) & 1);
                    plus = per || neu;
                    m = per ? T(0) : (neu ? L.h() : T(2));
                    off = per ? -o * n * stride : o * stride;
                    b = HB ? r[w.p + o * stride] : T(0);
                };
                side(0, ox, 1, L.nx, w.ox, w.mx, w.bx, w.nx);
                if (D == 3) side(1, oy, L.W, L.ny, w.oy, w.my, w.by, w.ny);
                side(D - 1, oz, L.PS, L.P, w.oz, w.mz, w.bz, w.nz);
                if (far) w.oz = -oz * L.P * L.PS;
            }
        }
        auto relax = [&](const CoCell<D, T, VAR> &w) {
            T *a = u + w.p;
            T val;
            if constexpr (VAR) {
                T x[2 * D], k[2 * D];
                co_neighbours<D, T>(a, L.W, L.PS, x);
#pragma unroll
                for (int s = 0; s < 2 * D; ++s) k[s] = w.c[s];
                val = var_quot<T>(var_dot<D, T>(k, x) + w.rs, w.c[2 * D], w.c[2 * D + 1]);
            } else {
                const T sum = D == 2 ? nb_sum6<D, T>(a[-1], a[1], a[-L.PS], a[L.PS], T(0), T(0))
                                     : nb_sum6<D, T>(a[-1], a[1], a[-L.W], a[L.W], a[-L.PS], a[L.PS]);
                val = fma(sum, inv, w.rs);
            }
            a[0] = val;
            if (w.ox) a[w.ox] = co_ghost_of<T, BC, HB>(w.mx, w.bx, w.nx, val);
            if (D == 3 && w.oy) a[w.oy] = co_ghost_of<T, BC, HB>(w.my, w.by, w.ny, val);
            if (w.oz) {
                if (far) co_store(far + (unsigned)sizeof(T) * (w.p + w.oz), val);
                else a[w.oz] = co_ghost_of<T, BC, HB>(w.mz, w.bz, w.nz, val);
            }
        };
        for (int half = 0; half < 2 * steps; ++half) {  // one copy of the body: its fetches count
            if (on) relax(c[0]);
            const CoCell<D, T, VAR> t = c[0];
            c[0] = c[1];
            c[1] = t;
            co_sync(L.nr);
        }
        return;
    }
    for (int sweep = 0; sweep < 2 * steps; ++sweep) {
        if (g < ng)
            for (int idx = first; idx < plane; idx += nt) {
                const int j = D == 3 ? co_div(idx, mh) : 0, x = idx - j * hx;
                for (int k = g; k < L.P; k += ng) {
                    const int i = 2 * x + ((sweep + j + L.z0 + k + D) & 1);
                    const int p = L.slot(i, j, k);
                    T val;
                    if constexpr (VAR) {
                        const int n = S.csz[li];
                        val = var_quot<T>(fma(-h2, r[p], co_dot<D, T>(cf + p, n, u + p, L.W, L.PS)),
                                          cf[2 * D * n + p], cf[(2 * D + 1) * n + p]);
                    } else {
                        const T sum = D == 2 ? nb_sum6<D, T>(u[p - 1], u[p + 1], u[p - L.PS], u[p + L.PS], T(0), T(0))
                                             : nb_sum6<D, T>(u[p - 1], u[p + 1], u[p - L.W], u[p + L.W], u[p - L.PS],
                                                             u[p + L.PS]);
                        val = fma(sum, inv, r[p] * chat);
                    }
                    co_put<D, T, BC, HB>(L, L.u, E, bc, p, i, j, k, val);
                }
            }
        co_sync(L.nr);
    }
}

// h^2 A u at slot p (FP64 adds, as in the per-level kernel of the coarse right-hand side)
template <int D, typename T, bool VAR>
__device__ __forceinline__ T co_lap(const CoarseArgs &S, const CoLevel<D, T> &L, int li, int p) {
    const T *u = co_mem<T>() + L.u;
    if constexpr (VAR) {
        const T *cf = co_mem<T>() + S.oc[li] + p;
        return fma(-cf[2 * D * S.csz[li]], u[p], co_dot<D, T>(cf, S.csz[li], u + p, L.W, L.PS));
    }
    if (D == 2) return nb_lap6<D, T, false>(u[p], u[p - 1], u[p + 1], u[p - L.PS], u[p + L.PS], T(0), T(0));
    return nb_lap6<D, T, false>(u[p], u[p - 1], u[p + 1], u[p - L.W], u[p + L.W], u[p - L.PS], u[p + L.PS]);
}

// Residual of level li restricted into level li - 1 (u and v' the mean of the
// children, then rho = I r + A u): Eq. residual and Eq. coarse-rhs.  When
// level li is spread over the blocks and li - 1 is not, every block stores
// its coarse values in all of them.
template <int D, typename T, bool BC, bool HB, bool VAR>
__device__ __noinline__ void co_down(int li, int rank, int bc) {
    const CoarseArgs &S = co_plan();
    T *sm = co_mem<T>();
    const CoLevel<D, T> L(li, rank), C(li - 1, rank);
    const bool spread = L.nr > 1 && C.nr == 1;
    const int Pc = L.P >> 1, zc = spread ? (L.z0 >> 1) : 0;  // coarse planes made here, first one in the coarse slab
    const unsigned mx = S.mx[li - 1], my = S.my[li - 1];
    const int n = C.nx * C.ny * Pc, nt = blockDim.x;
    const T ih2 = co_pow2<T>(2 * L.lg), ihc2 = co_pow2<T>(2 * C.lg), w = T(1) / T(1 << D);
    const bool wrap = BC && ((bc >> (6 + D - 1)) & 1);
    const CoEdge E = co_edge<T>(C.nr, rank, C.u, wrap);
    for (int c = threadIdx.x; c < n; c += nt) {
        int X, Y, Z;
        co_decode<D>(c, C.nx, mx, C.ny, my, X, Y, Z);
        T mu, rr;
        if constexpr (VAR) {
            const int nf = S.csz[li], rz = S.op == 2;
            const T *cf = sm + S.oc[li];
            T su = T(0), sr = T(0), sw = T(0);
#pragma unroll 1
            for (int q = 0; q < (1 << D); ++q) {
                const int i = 2 * X + (q & 1), j = D == 3 ? 2 * Y + ((q >> 1) & 1) : 0, k = 2 * Z + (q >> (D - 1));
                const int p = L.slot(i, j, k);
                const T uu = sm[L.u + p];
                const T lap = fma(-cf[2 * D * nf + p], uu, co_dot<D, T>(cf + p, nf, sm + L.u + p, L.W, L.PS));
                const T res = fma(-lap, ih2, sm[L.r + p]);
                const T wt = rz ? (T(i) + T(0.5)) * L.h() : T(1);
                su += wt * uu;
                sr += wt * res;
                sw += wt;
            }
            mu = rz ? su / sw : su * w;
            rr = rz ? sr / sw : sr * w;
        } else {
            T su = T(0), sro = T(0), sout = T(0);
            // sum_c (A u)_c = (sum_outside - D sum_c u) / h^2 over the 2^D children
#pragma unroll
            for (int dz = 0; dz < 2; ++dz)
#pragma unroll
                for (int dy = 0; dy < (D == 3 ? 2 : 1); ++dy)
#pragma unroll
                    for (int dx = 0; dx < 2; ++dx) {
                        const int p = L.slot(2 * X + dx, 2 * Y + dy, 2 * Z + dz);
                        const T *u = sm + L.u + p;
                        su += u[0];
                        sro += sm[L.r + p];
                        sout += u[dx ? 1 : -1];
                        if (D == 3) sout += u[dy ? L.W : -L.W];
                        sout += u[dz ? L.PS : -L.PS];
                    }
            mu = su * w;
            rr = fma(-ih2, fma(T(-D), su, sout), sro) * w;
        }
        const int k = zc + Z, p = C.slot(X, Y, k);
        sm[C.v + p] = mu;
        sm[C.r + p] = rr;
        if (!spread) {
            co_put<D, T, BC, HB>(C, C.u, E, bc, p, X, Y, k, mu);
        } else {
            for (int q = 0; q < S.R; ++q) {
                const unsigned base = co_map(sm, q) + (unsigned)sizeof(T) * p;
                co_store(base + (unsigned)sizeof(T) * C.u, mu);
                co_store(base + (unsigned)sizeof(T) * C.v, mu);
                co_store(base + (unsigned)sizeof(T) * C.r, rr);
            }
        }
    }
    co_sync(L.nr);
    const int nc = C.nx * C.ny * C.P;
    if (spread) {  // the ghosts of the whole grid, in every block
        for (int c = threadIdx.x; c < nc; c += nt) {
            int X, Y, Z;
            co_decode<D>(c, C.nx, mx, C.ny, my, X, Y, Z);
            const int p = C.slot(X, Y, Z);
            co_put<D, T, BC, HB>(C, C.u, E, bc, p, X, Y, Z, sm[C.u + p]);
        }
        __syncthreads();
    }
    for (int c = threadIdx.x; c < nc; c += nt) {
        int X, Y, Z;
        co_decode<D>(c, C.nx, mx, C.ny, my, X, Y, Z);
        const int p = C.slot(X, Y, Z);
        sm[C.r + p] = fma(ihc2, co_lap<D, T, VAR>(S, C, li - 1, p), sm[C.r + p]);
    }
    co_sync(C.nr);  // the next half-sweep stores halo values that this pass reads
}

// u += I (u_C - v'_C) from level li - 1, 2-1-1 (2D) / 1-1-1-1 (3D); across a
// domain side the difference is the homogeneous ghost of the cell inside.
template <int D, typename T, bool BC, bool HB>
__device__ __noinline__ void co_correct(int li, int rank, int bc) {
    const CoarseArgs &S = co_plan();
    T *sm = co_mem<T>();
    const CoLevel<D, T> L(li, rank), C(li - 1, rank);
    const int nt = blockDim.x, odc = S.odc;
    const bool wrap = BC && ((bc >> (6 + D - 1)) & 1);
    {
        const CoEdge E = co_edge<T>(C.nr, rank, odc, wrap);
        const int nc = C.nx * C.ny * C.P;
        const unsigned mx = S.mx[li - 1], my = S.my[li - 1];
        for (int c = threadIdx.x; c < nc; c += nt) {
            int X, Y, Z;
            co_decode<D>(c, C.nx, mx, C.ny, my, X, Y, Z);
            const int p = C.slot(X, Y, Z);
            co_put<D, T, BC, false>(C, odc, E, bc, p, X, Y, Z, sm[C.u + p] - sm[C.v + p]);
        }
    }
    co_sync(C.nr);
    const CoEdge E = co_edge<T>(L.nr, rank, L.u, wrap);
    const int n = L.nx * L.ny * L.P;
    const unsigned mx = S.mx[li], my = S.my[li];
    for (int c = threadIdx.x; c < n; c += nt) {
        int i, j, k;
        co_decode<D>(c, L.nx, mx, L.ny, my, i, j, k);
        const int kz = L.z0 + k;
        const T *d = sm + odc + C.slot(i >> 1, j >> 1, (kz >> 1) - C.z0);
        const T d0 = d[0], dx = d[(i & 1) ? 1 : -1], dz = d[(kz & 1) ? C.PS : -C.PS];
        const int p = L.slot(i, j, k);
        T val;
        if (D == 2) {
            val = fma(T(0.25), dx + dz, fma(T(0.5), d0, sm[L.u + p]));
        } else {
            const T dy = d[(j & 1) ? C.W : -C.W];
            val = fma(T(0.25), ((d0 + dx) + dy) + dz, sm[L.u + p]);
        }
        co_put<D, T, BC, HB>(L, L.u, E, bc, p, i, j, k, val);
    }
    co_sync(L.nr);
}

template <int D, typename T, bool BC, bool HB, bool VAR>
__device__ __noinline__ void co_vcycle(int lt, int rank, int bc) {
    const CoarseArgs &S = co_plan();
    for (int li = lt; li > 0; --li) {
        co_smooth<D, T, BC, HB, VAR>(li, S.nd, rank, bc);
        co_down<D, T, BC, HB, VAR>(li, rank, bc);
    }
    co_smooth<D, T, BC, HB, VAR>(0, S.nb, rank, bc);
    for (int li = 1; li <= lt; ++li) {
        co_correct<D, T, BC, HB>(li, rank, bc);
        co_smooth<D, T, BC, HB, VAR>(li, S.nu, rank, bc);
    }
}

// Calls f(s, i, j, k, ghost slot, t1, t2) for every face cell of this block's
// part of a level's domain sides (periodic axes have none): (i, j, k) the cell
// inside (local plane k), (t1, t2) its tangential indices over the whole
// grid, x first.
template <int D, typename T, typename F>
__device__ __forceinline__ void co_faces(const CoLevel<D, T> &L, int rank, int bc, F f) {
    const int last = D - 1;
    for (int s = 0; s < 2 * D; ++s) {
        const int a = s >> 1, up = s & 1;
        if ((bc >> (6 + a)) & 1) continue;
        if (a == last && L.nr > 1 && rank != (up ? L.nr - 1 : 0)) continue;
        const int n1 = a == 0 ? (D == 3 ? L.ny : L.P) : L.nx;  // local extent of the first tangential axis
        const int n2 = D == 2 ? 1 : (a == last ? L.ny : L.P);
        for (int e = threadIdx.x; e < n1 * n2; e += blockDim.x) {
            const int e2 = e / n1, e1 = e - e2 * n1;
            int i, j = 0, k;
            if (a == 0) {
                i = up ? L.nx - 1 : 0;
                j = D == 3 ? e1 : 0;
                k = D == 3 ? e2 : e1;
            } else if (a == last) {
                i = e1;
                j = D == 3 ? e2 : 0;
                k = up ? L.P - 1 : 0;
            } else {
                i = e1;
                j = up ? L.ny - 1 : 0;
                k = e2;
            }
            const int step = a == 0 ? 1 : (a == last ? L.PS : L.W);
            f(s, i, j, k, L.slot(i, j, k) + (up ? step : -step));
        }
    }
}

// mean of the 2^(D-1) boundary values of level F under the face of cell
// (i, j, k) on side s of the next coarser level (k and F's planes local)
template <int D, typename T>
__device__ __forceinline__ T co_face_mean(const CoLevel<D, T> &F, int s, int i, int j, int k) {
    const T *r = co_mem<T>() + F.r;
    const int a = s >> 1, up = s & 1, last = D - 1;
    const int step = a == 0 ? 1 : (a == last ? F.PS : F.W);
    T sum = T(0);
    for (int e2 = 0; e2 < (D == 3 ? 2 : 1); ++e2)
        for (int e1 = 0; e1 < 2; ++e1) {
            const int fi = 2 * i + (a == 0 ? up : e1);
            const int fj = D == 3 ? 2 * j + (a == 1 ? up : (a == 0 ? e1 : e2)) : 0;
            const int fk = 2 * k + (a == last ? up : (D == 3 ? e2 : e1));
            sum += r[F.slot(fi, fj, fk) + (up ? step : -step)];
        }
    return sum * (T(1) / T(1 << (D - 1)));
}

// Boundary data of every level held here, for the ghost slots of the sources:
// level top's from the boxes, below it the mean of the 2^(D-1) finer faces.
// Gathered once per change of the data (mode 2), not in every cycle: the
// gather costs 17 us, reading its result one load per face.
template <int D, typename T>
__device__ __noinline__ void co_gather_faces(const BoxMeta &A, int rank, int bc, double *fval) {
    const CoarseArgs &S = co_plan();
    T *sm = co_mem<T>();
    const int tid = threadIdx.x, nt = blockDim.x, lt = S.nl - 1, mb = S.mb, lg = S.lgmb;
    const CoLevel<D, T> L(lt, rank);
    const int *dbox = S.dbox + (size_t)(blockIdx.x / S.R) * S.nbx * S.nby * S.nbz;
    co_faces<D, T>(L, rank, bc, [&](int s, int i, int j, int k, int gs) {
        const int kz = L.z0 + k, a = s >> 1, m1 = mb - 1, jj = D == 3 ? j : kz, kk = D == 3 ? kz : 0;
        const int b = dbox[((kk >> lg) * S.nby + (jj >> lg)) * S.nbx + (i >> lg)];
        const int f1 = (a == 0 ? jj : i) & m1, f2 = D == 3 ? (a == 2 ? j : kz) & m1 : 0;
        sm[L.r + gs] = T(A.bc[A.nbase[b * 2 * D + s] + f2 * mb + f1]);
    });
    for (int li = lt - 1; li >= 0; --li) {
        const CoLevel<D, T> F(li + 1, rank), B(li, rank);
        __syncthreads();
        if (F.nr > 1 && B.nr == 1) {
            // held whole by every block: each stores the faces above its planes in all of them
            CoLevel<D, T> V = B;  // the coarse planes over this block's slab
            V.P = F.P >> 1;
            V.nr = F.nr;
            const int zc = F.z0 >> 1;
            co_faces<D, T>(V, rank, bc, [&](int s, int i, int j, int k, int gs) {
                const T b = co_face_mean<D, T>(F, s, i, j, k);
                for (int q = 0; q < S.R; ++q) co_store(co_map(sm, q) + (unsigned)sizeof(T) * (B.r + gs + zc * B.PS), b);
            });
            co_cluster_sync();
        } else {
            co_faces<D, T>(B, rank, bc, [&](int s, int i, int j, int k, int gs) {
                sm[B.r + gs] = co_face_mean<D, T>(F, s, i, j, k);
            });
        }
    }
    __syncthreads();
    const int at = (blockIdx.x / S.R * S.R + rank) * S.nface;
    for (int x = tid; x < S.nface; x += nt) {
        const int q = S.fslot[rank * S.nface + x];
        if (q >= 0) fval[at + x] = (double)sm[q];
    }
}

// The coefficients of every level held here, packed in the layout of this
// block's shared memory (mode 3, after eps changed).
template <int D, typename T>
__device__ __noinline__ void co_gather_coef(const BoxMeta &A, int rank, T *cpack) {
    const CoarseArgs &S = co_plan();
    T *out = cpack + (size_t)(blockIdx.x / S.R * S.R + rank) * S.ncoef;
    const int tree = blockIdx.x / S.R;
    for (int li = 0; li < S.nl; ++li) {
        const CoLevel<D, T> L(li, rank);
        int lg = 0;  // cells per box side
        while ((2 << lg) <= S.N && lg <= li) ++lg;
        const int mb = 1 << lg, nbx = L.nx >> lg, nby = (D == 3 ? L.ny : L.P * L.nr) >> lg;
        const int nbz = D == 3 ? (L.P * L.nr) >> lg : 1, H = (D == 2 ? mb * mb : mb * mb * mb) / 2;
        for (int c = threadIdx.x; c < L.nx * L.ny * L.P; c += blockDim.x) {
            int i, j, k;
            co_decode<D>(c, L.nx, S.mx[li], L.ny, S.my[li], i, j, k);
            const int kz = L.z0 + k, jj = D == 3 ? j : kz, kk = D == 3 ? kz : 0, m1 = mb - 1;
            const int b = S.dtab[li][((size_t)tree * nbz + (kk >> lg)) * nby * nbx + (jj >> lg) * nbx + (i >> lg)];
            const long long q = A.coff[b] + ((i + j + kz + D) & 1) * H + ((kk & m1) * mb + (jj & m1)) * (mb / 2) +
                                ((i & m1) >> 1);
            for (int f = 0; f < 2 * D + 2; ++f)
                out[S.oc[li] - S.ocoef + f * S.csz[li] + L.slot(i, j, k)] =
                    reinterpret_cast<const T *>(S.coef)[f * S.coef_n + q];
        }
    }
}

template <int D, typename T, bool BC, bool HB, bool VAR>
__device__ __forceinline__ void co_run(int rank, int bc, const long long *cell0, const unsigned char *refined, T *u,
                                       const T *rho, T *vold) {
    const CoarseArgs &S = co_plan();
    T *sm = co_mem<T>();
    const int tid = threadIdx.x, nt = blockDim.x, lt = S.nl - 1, mb = S.mb, lg = S.lgmb;
    const CoLevel<D, T> L(lt, rank);
    const CoEdge E = co_edge<T>(L.nr, rank, L.u, BC && ((bc >> (6 + D - 1)) & 1));
    const int half = L.nx >> 1, n = half * L.ny * L.P, H = (D == 2 ? mb * mb : mb * mb * mb) / 2;
    const unsigned mh = S.mh[lt], my = S.my[lt];
    const int b0 = D == 3 ? (L.z0 >> lg) * S.nby * S.nbx : (L.z0 >> lg) * S.nbx;  // first box of the slab's table
    // half-row position c -> its first cell (x = 2h), box in the slab's table, cell offset in the box (red half)
    auto where = [&](int c, int &x, int &j, int &k, int &box, int &at, int &r0) {
        co_decode<D>(c, half, mh, L.ny, my, x, j, k);
        const int kz = L.z0 + k;
        const int bx = (2 * x) >> lg, jj = D == 3 ? j : kz, kk = D == 3 ? kz : 0;
        box = ((kk >> lg) * S.nby + (jj >> lg)) * S.nbx + bx - b0;
        at = ((kk & (mb - 1)) * mb + (jj & (mb - 1))) * (mb / 2) + (x & (mb / 2 - 1));
        r0 = (j + kz + D) & 1;  // red cell at 2x + r0
    };
    if constexpr (VAR) {  // the packed coefficients, waited for before the first use
        const char *src = reinterpret_cast<const char *>(S.cpack) +
                          (size_t)(blockIdx.x / S.R * S.R + rank) * S.ncoef * sizeof(T);
        char *dst = reinterpret_cast<char *>(sm + S.ocoef);
        for (int x = tid; x < (int)(S.ncoef * sizeof(T) / 16); x += nt) cp_async<16>(dst + 16 * x, src + 16 * x);
        cp_commit();
    }
    constexpr int Q = 4;  // loads of a batch are in flight together
    for (int c0 = tid; c0 < n; c0 += Q * nt) {
        T ur[Q], ub[Q], rr[Q], rb[Q];
        int p[Q], r0[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int c = c0 + q * nt;
            if (c >= n) break;
            int x, j, k, box, at;
            where(c, x, j, k, box, at, r0[q]);
            const long long g = cell0[box] + at;
            p[q] = L.slot(2 * x, j, k);
            ur[q] = u[g];
            ub[q] = u[g + H];
            rr[q] = rho[g];
            rb[q] = rho[g + H];
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (c0 + q * nt >= n) break;
            sm[L.r + p[q] + r0[q]] = rr[q];
            sm[L.r + p[q] + 1 - r0[q]] = rb[q];
            sm[L.u + p[q] + r0[q]] = ur[q];
            sm[L.u + p[q] + 1 - r0[q]] = ub[q];
        }
    }
    if (HB) {  // boundary data into the ghost slots of the sources
        const int at = (blockIdx.x / S.R * S.R + rank) * S.nface;
        for (int x = tid; x < S.nface; x += nt) {
            const int q = S.fslot[rank * S.nface + x];
            if (q >= 0) sm[q] = T(S.fval[at + x]);
        }
    }
    if constexpr (VAR) cp_wait<0>();
    __syncthreads();
    for (int c = tid; c < n; c += nt) {  // ghosts and halos of level top's solution
        int x, j, k;
        co_decode<D>(c, half, mh, L.ny, my, x, j, k);
        const int p = L.slot(2 * x, j, k);
        co_put<D, T, BC, HB>(L, L.u, E, bc, p, 2 * x, j, k, sm[L.u + p]);
        co_put<D, T, BC, HB>(L, L.u, E, bc, p + 1, 2 * x + 1, j, k, sm[L.u + p + 1]);
    }
    co_sync(L.nr);
    if (S.fas) {
        const T ih2 = co_pow2<T>(2 * L.lg);
        for (int c = tid; c < n; c += nt) {
            int x, j, k, box, at, r0;
            where(c, x, j, k, box, at, r0);
            const int p = L.slot(2 * x, j, k);
            if (refined[box]) {
                sm[L.r + p] = fma(ih2, co_lap<D, T, VAR>(S, L, lt, p), sm[L.r + p]);
                sm[L.r + p + 1] = fma(ih2, co_lap<D, T, VAR>(S, L, lt, p + 1), sm[L.r + p + 1]);
            } else {
                const long long g = cell0[box] + at;
                vold[g] = sm[L.u + p + r0];
                vold[g + H] = sm[L.u + p + 1 - r0];
            }
        }
        co_sync(L.nr);
    }
    if (S.mode == 0) {
        co_vcycle<D, T, BC, HB, VAR>(lt, rank, bc);
    } else {
        for (int li = lt; li > 0; --li) co_down<D, T, BC, HB, VAR>(li, rank, bc);
        for (int li = 0; li <= lt; ++li) {
            const CoLevel<D, T> B(li, rank);
            if (li < lt) {
                const int np = (B.P + 2) * B.PS;
                for (int p = tid; p < np; p += nt) sm[B.v + p] = sm[B.u + p];
            } else {
                for (int c = tid; c < n; c += nt) {
                    int x, j, k, box, at, r0;
                    where(c, x, j, k, box, at, r0);
                    const long long g = cell0[box] + at;
                    const int p = L.slot(2 * x, j, k);
                    vold[g] = sm[L.u + p + r0];
                    vold[g + H] = sm[L.u + p + 1 - r0];
                }
            }
            __syncthreads();
            if (li > 0) co_correct<D, T, BC, HB>(li, rank, bc);
            co_vcycle<D, T, BC, HB, VAR>(li, rank, bc);
        }
    }
    if (rank == 0 || L.nr > 1)
        for (int c = tid; c < n; c += nt) {
            int x, j, k, box, at, r0;
            where(c, x, j, k, box, at, r0);
            const long long g = cell0[box] + at;
            const int p = L.slot(2 * x, j, k);
            u[g] = sm[L.u + p + r0];
            u[g + H] = sm[L.u + p + 1 - r0];
        }
}

// grid: R blocks (one cluster) per tree.  mode 0: V-cycle from level top;
// mode 1: restriction of level top's values to the coarsest grid with the
// coarse right-hand sides, then the FMG steps up to level top (v'_l <- v_l,
// correction from l - 1, V-cycle from l), level top's v' going to global
// memory; mode 2: the boundary data of the levels gathered into G.fval (after
// it changed); mode 3 (VAR): the coefficients packed into G.cpack (after eps
// changed).  fas: level top's source holds the restricted residual; its coarse
// right-hand side rho + A u is completed here (refined boxes), and its leaf
// boxes store v' = u.
template <int D, typename T, bool VAR>
__global__ void __launch_bounds__(kCoarseThreads) k_coarse(BoxMeta A, const __grid_constant__ CoarseArgs G, T *u,
                                                           const T *rho, T *vold) {
    const int rank = G.R > 1 ? (int)(blockIdx.x % G.R) : 0, tree = blockIdx.x / G.R;
    const int tid = threadIdx.x, nt = blockDim.x;
    pdl_trigger();
    // before the wait: the plan, the boxes of this block's slab, zeros in the
    // source's ghost slots (homogeneous boundary data)
    for (int x = tid; x < (int)(sizeof(CoarseArgs) / 4); x += nt)
        reinterpret_cast<int *>(co_smem)[x] = reinterpret_cast<const int *>(&G)[x];
    T *sm = co_mem<T>();
    const int grids = VAR ? G.ocoef : G.total;
    for (int x = tid; x < grids; x += nt) sm[x] = T(0);
    const int lt = G.nl - 1, z0 = G.nr[lt] > 1 ? rank * G.P[lt] : 0;
    const int layer = D == 3 ? G.nbx * G.nby : G.nbx;
    const int first = (z0 >> G.lgmb) * layer, nbox = (((z0 + G.P[lt] - 1) >> G.lgmb) + 1) * layer - first;
    long long *cell0 =
        reinterpret_cast<long long *>(co_smem + kCoarseHead + ((size_t)G.total * sizeof(T) + 15) / 16 * 16);
    unsigned char *refined = reinterpret_cast<unsigned char *>(cell0 + G.slab_boxes);
    const int *dbox = G.dbox + (size_t)tree * G.nbx * G.nby * G.nbz;
    for (int x = tid; x < nbox; x += nt) {
        const int b = dbox[first + x];
        cell0[x] = A.coff[b];
        refined[x] = A.bflag[b] & BF_REFINED;
    }
    const int bc = G.tree_bc[tree];
    __syncthreads();
    pdl_wait();
    if (A.active && !A.active[tree]) return;  // R = 1 here: no barrier of a cluster is skipped
    if (G.R > 1) co_cluster_sync();           // every block has cleared its memory before another stores into it
    if (G.mode == 2) co_gather_faces<D, T>(A, rank, bc, G.fval);
    else if (VAR && G.mode == 3) co_gather_coef<D, T>(A, rank, reinterpret_cast<T *>(G.cpack));
    else if (bc) {
        if (G.hom) co_run<D, T, true, false, VAR>(rank, bc, cell0, refined, u, rho, vold);
        else co_run<D, T, true, true, VAR>(rank, bc, cell0, refined, u, rho, vold);
    } else {
        if (G.hom) co_run<D, T, false, false, VAR>(rank, bc, cell0, refined, u, rho, vold);
        else co_run<D, T, false, true, VAR>(rank, bc, cell0, refined, u, rho, vold);
    }
    if (G.R > 1) co_cluster_sync();  // no block leaves while another may store into it
}

}  // namespace afg
