// Red-black Gauss-Seidel half-sweep (Sec. 3.1 of arXiv:1701.04329) with a
// half-row shared-memory layout and cp.async staging, for boxes whose colour
// half-rows hold at least one 16-byte vector (M/2 >= 16/sizeof(T)).  The
// other boxes (2 cells per side, and 4 in FP32) take the table-driven k_smooth.
//
// A half-sweep of colour c reads only cells of colour 1-c.  In a row (j,k)
// the cells of one colour sit at i = 2h + r with r fixed per row, so the
// colour 1-c cells of a box plus the ghost cells a colour-c update reads form
// an array of half-rows P[k+1][j+1][h], h in [0, M/2), rows j, k in [-1, M],
// plus the x-side ghosts X[side][row].  For the VEC colour-c cells
// h0..h0+VEC-1 of row (j,k), with r = (c+j+k+D) & 1:
//   y and z neighbours: half-rows (j+-1,k), (j,k+-1) at h0..h0+VEC-1 (in those
//   rows the colour 1-c cells sit at the same i);
//   x neighbours: half-row (j,k) at h0+r-1 .. h0+r+VEC-1 (one vector and one
//   scalar, the scalar from X at the ends of the row).
//
// The colour 1-c half-rows, the colour-c source values and the ghost layer of
// a box are copied global -> shared with cp.async into a ring of NST stages,
// so the copies of the next box of a group are in flight while the current
// one is relaxed.  Same-level ghosts are plain copies of the neighbour's
// half-rows (y, z sides) or values (x sides).  Ghosts of domain-boundary and
// refinement-boundary faces are staged as the adjacent inner value u_1 and
// completed after the wait: g = 2b - u_1 (Dirichlet) or
// g = u_H/2 + c1 u_1 - (u_2 + u_t1 [+ u_t2])/4 (Sec. 3.3).  Within a colour-c
// half-sweep no box writes what another box's copies read (colour 1-c
// halves, coarse data, the box's own colour-c half before its own update),
// so staging ahead is safe.
#pragma once
#include "kernels.cuh"

namespace afg {

// storage offset, inside a colour half, of the half-row (j,k)
template <int D, int M>
__device__ __forceinline__ int hrow(int j, int k) { return (k * M + j) * (M / 2); }

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(BYTES)
                     : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Metadata of entry `idx` of a level range or list into slot I, asynchronously:
// the box's BoxInfo in 16-byte pieces.  (Thirteen loads whose results a thread
// then stored made the first warp of every box's group wait for L2 ahead of
// the box's arithmetic: 256^3, half-sweeps FP64 72.2 -> 64.4 us, FP32 23.5 -> 21.1
// us, FP64 restriction 165 -> 148 us; uniform 512^3, mixed, 49.2 -> 44.7 ms; 128
// masked quadtrees, mixed, 16.8 -> 15.5 ms.)  Done after the thread's next cp_wait
// and a barrier.
template <int D>
__device__ __forceinline__ void info_stage(const BoxMeta &A, int idx, int n, int b0, const int *list, BoxInfo &I,
                                           int lt, int G) {
    constexpr int NP = (int)sizeof(BoxInfo) / 16;
    if (idx >= n) {
        if (lt == 0) I.b = -1;
        return;
    }
    if (lt >= NP) return;
    const char *src = reinterpret_cast<const char *>(A.info + (list ? list[idx] : b0 + idx));
    for (int x = lt; x < NP; x += G) cp_async<16>(reinterpret_cast<char *>(&I) + 16 * x, src + 16 * x);
}

// whether a staged slot holds a box of a tree that takes part (the mask stays in
// L1; the walks ask where they stage a box and where they compute it)
__device__ __forceinline__ bool info_on(const BoxMeta &A, const BoxInfo &I) {
    return I.b >= 0 && (!A.active || A.active[I.tree]);
}

// VPT: 16-byte vectors of a box's colour half per thread (1: one thread per
// vector; 2: half as many threads per box, twice the boxes per CTA)
template <int D, int M, typename T, int VPT = 1>
struct SpCfg {
    static constexpr int VEC = 16 / (int)sizeof(T);
    static constexpr int MH = M / 2;
    static constexpr int ROWS = D == 2 ? (M + 2) : (M + 2) * (M + 2);
    static constexpr int PT = ROWS * MH;     // colour 1-c half-rows, interior and y/z ghost rows
    static constexpr int XT = 2 * ROWS;      // x-side ghosts [side][row]
    static constexpr int H = Geo<D, M>::H;
    static constexpr int BOX = PT + XT + H;  // + colour-c source values
    static constexpr int NVR = MH / VEC;
    static constexpr int FR = D == 2 ? 1 : M;
    static constexpr int NV = H / VEC;
    static constexpr int G = (NV / VPT > 0 ? NV / VPT : 1) < kThreads ? (NV / VPT > 0 ? NV / VPT : 1) : kThreads;
    static constexpr int BPC = kThreads / G;
    static constexpr int NIT = (NV + G - 1) / G;
    static constexpr int NXI = (D == 2 ? M : M * M) / 2;
    static constexpr int NGI = 2 * NXI + (2 * D - 2) * FR * NVR;
    static constexpr int NST = 2;  // more stages cost resident CTAs and measured slower
    static constexpr size_t smem() { return sizeof(T) * BOX * BPC * NST + sizeof(BoxInfo) * BPC * (NST + 1); }
    static constexpr bool ok = MH >= VEC;
};

// padded row of (j,k), ghost rows included
template <int D, int M>
__device__ __forceinline__ int sp_row(int j, int k) { return D == 2 ? (j + 1) : (k + 1) * (M + 2) + (j + 1); }

// x-side ghost item -> side and row (rows whose colour-c cell touches side s)
template <int D, int M>
__device__ __forceinline__ void sp_xitem(int item, int c, int &s, int &j, int &k) {
    constexpr int MH = M / 2, NXI = (D == 2 ? M : M * M) / 2;
    s = item / NXI;
    const int ri = item % NXI;
    if (D == 2) { k = 0; j = 2 * ri + ((s + c + D) & 1); }
    else { k = ri / MH; j = 2 * (ri % MH) + ((s + c + k + D) & 1); }
}

// y/z-side ghost item -> side, vector start, ghost row, inner row, mirror row in the neighbour
template <int D, int M, typename T>
__device__ __forceinline__ void sp_yzitem(int it2, int &s, int &h0, int &jg, int &kg, int &jin, int &kin, int &jm,
                                          int &km) {
    using S = SpCfg<D, M, T>;
    s = 2 + it2 / (S::FR * S::NVR);
    const int rem = it2 % (S::FR * S::NVR);
    const int fr = rem / S::NVR;
    h0 = (rem % S::NVR) * S::VEC;
    const int hi = s & 1;
    if ((s >> 1) == 1) { kg = kin = km = D == 3 ? fr : 0; jg = hi ? M : -1; jin = hi ? M - 1 : 0; jm = hi ? 0 : M - 1; }
    else { jg = jin = jm = fr; kg = hi ? M : -1; kin = hi ? M - 1 : 0; km = hi ? 0 : M - 1; }
}

// Per-thread copy plan, the same for every box of a launch (fixed colour):
// for each ghost item of the thread, the destination in the box's stage, the
// side, whether it is a scalar (x side), and the source offsets relative to
// the neighbour box (same-level copy) and to the box's own colour-c half (u_1).
template <int D, int M, typename T, int VPT = 1>
struct SpPlan {
    using S = SpCfg<D, M, T, VPT>;
    static constexpr int NQ = (S::NGI + S::G - 1) / S::G;
    int gdst[NQ], gsrc[NQ];  // dst | side << 16 | scalar << 19 ; nb offset | u1 offset << 16
    int gbc[NQ];             // boundary data of the item's first face (stride 2 along a y/z item's vector)
    int vdst[S::NIT], vsrc[S::NIT];
    __device__ __forceinline__ void init(int lt, int c) {
        constexpr int MH = S::MH, H = S::H;
#pragma unroll
        for (int it = 0; it < S::NIT; ++it) {
            const int v = lt + it * S::G;
            const int row = v / S::NVR, h0 = (v % S::NVR) * S::VEC;
            const int j = row % M, k = D == 2 ? 0 : row / M;
            vdst[it] = v < S::NV ? sp_row<D, M>(j, k) * MH + h0 : -1;
            vsrc[it] = hrow<D, M>(j, k) + h0;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int item = lt + q * S::G;
            gdst[q] = -1;
            gsrc[q] = 0;
            gbc[q] = 0;
            if (item >= S::NGI) continue;
            if (item < 2 * S::NXI) {
                int sd, j, k;
                sp_xitem<D, M>(item, c, sd, j, k);
                gbc[q] = k * M + j;
                gdst[q] = (S::PT + sd * S::ROWS + sp_row<D, M>(j, k)) | (sd << 16) | (1 << 19);
                gsrc[q] = ((1 - c) * H + hrow<D, M>(j, k) + (sd ? 0 : MH - 1)) | ((hrow<D, M>(j, k) + (sd ? MH - 1 : 0)) << 16);
            } else {
                int sd, h0, jg, kg, jin, kin, jm, km;
                sp_yzitem<D, M, T>(item - 2 * S::NXI, sd, h0, jg, kg, jin, kin, jm, km);
                const int rg = (c + jin + kin + D) & 1;  // i-parity of the colour-c cells of the inner row
                gbc[q] = ((sd >> 1) == 1 ? kin : jin) * M + 2 * h0 + rg;
                gdst[q] = (sp_row<D, M>(jg, kg) * MH + h0) | (sd << 16);
                gsrc[q] = ((1 - c) * H + hrow<D, M>(jm, km) + h0) | ((hrow<D, M>(jin, kin) + h0) << 16);
            }
        }
    }
};

template <int D, int M, typename T, int VPT>
__device__ __forceinline__ void sp_issue(const SpPlan<D, M, T, VPT> &pl, const BoxInfo &I, const T *u, const T *rho,
                                         T *box, int lt, int c) {
    using S = SpCfg<D, M, T, VPT>;
    constexpr int VEC = S::VEC, H = S::H;
    const T *uo = u + I.coff + (1 - c) * H, *uc = u + I.coff + c * H;
    T *R = box + S::PT + S::XT;
#pragma unroll
    for (int it = 0; it < S::NIT; ++it) {
        const int v = lt + it * S::G;
        if (v >= S::NV) continue;
        cp_async<16>(box + pl.vdst[it], uo + pl.vsrc[it]);
        cp_async<16>(R + v * VEC, rho + I.coff + c * H + v * VEC);
    }
#pragma unroll
    for (int q = 0; q < SpPlan<D, M, T, VPT>::NQ; ++q) {
        const int dst = pl.gdst[q];
        if (dst < 0) continue;
        const int sd = (dst >> 16) & 7;
        const T *src = I.code[sd] >= 0 ? u + I.base[sd] + (pl.gsrc[q] & 0xffff) : uc + (pl.gsrc[q] >> 16);
        if (dst & (1 << 19)) cp_async<(int)sizeof(T)>(box + (dst & 0xffff), src);
        else cp_async<16>(box + (dst & 0xffff), src);
    }
}

// Completes the domain-side ghosts among this thread's own items from the
// u_1 it staged there (visible to it after its own wait, before the box's
// barrier): 2 b - u_1 (Dirichlet) or u_1 + h b (Neumann).
template <int D, int M, typename T, int VPT>
__device__ __forceinline__ void sp_fix_own(const SpPlan<D, M, T, VPT> &pl, const BoxInfo &I, const BoxMeta &A, T *box,
                                           int hom) {
    using S = SpCfg<D, M, T, VPT>;
    constexpr int VEC = S::VEC;
#pragma unroll
    for (int q = 0; q < SpPlan<D, M, T, VPT>::NQ; ++q) {
        const int dst = pl.gdst[q];
        if (dst < 0) continue;
        const int sd = (dst >> 16) & 7;
        if (I.code[sd] != -1) continue;
        const bool neu = (I.nmask >> sd) & 1;
        const T hbox = neu ? T(A.hb[I.b]) : T(0);
        const double *bc = A.bc + I.base[sd] + pl.gbc[q];
        T *gv = box + (dst & 0xffff);
        if (dst & (1 << 19)) {
            const T bv = hom ? T(0) : T(bc[0]);
            gv[0] = neu ? fma(hbox, bv, gv[0]) : T(2) * bv - gv[0];
        } else {
#pragma unroll
            for (int x = 0; x < VEC; ++x) {
                const T bv = hom ? T(0) : T(bc[2 * x]);
                gv[x] = neu ? fma(hbox, bv, gv[x]) : T(2) * bv - gv[x];
            }
        }
    }
}

// completes the ghosts of non-copy faces from the staged u_1 (cf_only: the
// refinement-boundary faces only, the domain sides being done by sp_fix_own)
template <int D, int M, typename T, int VPT = 1>
__device__ __forceinline__ void sp_fix(const BoxInfo &I, const BoxMeta &A, const T *u, T *box, int lt, int c,
                                       int hom, bool cf_only = false) {
    using S = SpCfg<D, M, T, VPT>;
    constexpr int VEC = S::VEC, MH = S::MH;
    T *P = box, *X = box + S::PT;
    const T c1 = D == 2 ? T(1) : T(1.25);
    // interior cell (i,j,k) of colour 1-c
    auto at = [&](int i, int j, int k) -> T { return P[sp_row<D, M>(j, k) * MH + (i >> 1)]; };
    for (int item = lt; item < S::NGI; item += S::G) {
        if (item < 2 * S::NXI) {
            int s, j, k;
            sp_xitem<D, M>(item, c, s, j, k);
            const int code = I.code[s];
            if (code >= 0 || (cf_only && code == -1)) continue;
            T &gv = X[s * S::ROWS + sp_row<D, M>(j, k)];
            const T u1 = gv;
            if (code == -1) {
                if ((I.nmask >> s) & 1) continue;  // Neumann: the pass below
                const T bv = hom ? T(0) : T(A.bc[I.base[s] + k * M + j]);
                gv = T(2) * bv - u1;
            } else {
                const int iin = s ? M - 1 : 0, p2 = s ? M - 2 : 1;
                const int cj = unpack_off(I.poff, 1) + (j >> 1);
                const int ck = D == 3 ? unpack_off(I.poff, 2) + (k >> 1) : 0;
                const T uH = u[I.base[s] + rbi<D, M>(s ? 0 : M - 1, cj, ck)];
                T acc = at(p2, j, k) + at(iin, j ^ 1, k);
                if (D == 3) acc += at(iin, j, k ^ 1);
                gv = T(0.5) * uH + c1 * u1 - T(0.25) * acc;
            }
        } else {
            int s, h0, jg, kg, jin, kin, jm, km;
            sp_yzitem<D, M, T>(item - 2 * S::NXI, s, h0, jg, kg, jin, kin, jm, km);
            const int code = I.code[s];
            if (code >= 0 || (cf_only && code == -1)) continue;
            const int hi = s & 1, a = s >> 1;
            T *gv = P + sp_row<D, M>(jg, kg) * MH + h0;
            const int rg = (c + jin + kin + D) & 1;  // i-parity of the colour-c cells of the inner row
            const int p2 = hi ? M - 2 : 1;
#pragma unroll
            for (int x = 0; x < VEC; ++x) {
                const int i = 2 * (h0 + x) + rg;
                const T u1 = gv[x];
                if (code == -1) {
                    const int t2 = a == 1 ? kin : jin;
                    if ((I.nmask >> s) & 1) continue;  // Neumann: the pass below
                    const T bv = hom ? T(0) : T(A.bc[I.base[s] + t2 * M + i]);
                    gv[x] = T(2) * bv - u1;
                } else {
                    const int ci = unpack_off(I.poff, 0) + (i >> 1);
                    int cj, ck;
                    T acc;
                    if (a == 1) {
                        cj = hi ? 0 : M - 1;
                        ck = D == 3 ? unpack_off(I.poff, 2) + (kin >> 1) : 0;
                        acc = at(i, p2, kin) + at(i ^ 1, jin, kin);
                        if (D == 3) acc += at(i, jin, kin ^ 1);
                    } else {
                        cj = unpack_off(I.poff, 1) + (jin >> 1);
                        ck = hi ? 0 : M - 1;
                        acc = at(i, jin, p2) + at(i ^ 1, jin, kin);
                        acc += at(i, jin ^ 1, kin);
                    }
                    const T uH = u[I.base[s] + rbi<D, M>(ci, cj, ck)];
                    gv[x] = T(0.5) * uH + c1 * u1 - T(0.25) * acc;
                }
            }
        }
    }
    if (!I.nmask || cf_only) return;
    // Neumann domain sides: g = u_1 + h b (a separate pass keeps the common path lean)
    const T hbox = T(A.hb[I.b]);
    for (int item = lt; item < S::NGI; item += S::G) {
        if (item < 2 * S::NXI) {
            int s, j, k;
            sp_xitem<D, M>(item, c, s, j, k);
            if (I.code[s] != -1 || !((I.nmask >> s) & 1)) continue;
            T &gv = X[s * S::ROWS + sp_row<D, M>(j, k)];
            const T bv = hom ? T(0) : T(A.bc[I.base[s] + k * M + j]);
            gv = fma(hbox, bv, gv);
        } else {
            int s, h0, jg, kg, jin, kin, jm, km;
            sp_yzitem<D, M, T>(item - 2 * S::NXI, s, h0, jg, kg, jin, kin, jm, km);
            if (I.code[s] != -1 || !((I.nmask >> s) & 1)) continue;
            T *gv = P + sp_row<D, M>(jg, kg) * MH + h0;
            const int rg = (c + jin + kin + D) & 1;
            const int t2 = (s >> 1) == 1 ? kin : jin;
#pragma unroll
            for (int x = 0; x < VEC; ++x) {
                const int i = 2 * (h0 + x) + rg;
                const T bv = hom ? T(0) : T(A.bc[I.base[s] + t2 * M + i]);
                gv[x] = fma(hbox, bv, gv[x]);
            }
        }
    }
}

// barrier of one box's thread group (g: its number in the block).  The barrier
// numbers are constants: with one in a register a block reserves all 16, and an
// SM holds four such blocks at most.
template <int G, int X = 0>
__device__ __forceinline__ void group_sync(int g) {
    if constexpr (G <= 32) {
        __syncwarp(G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1) << ((threadIdx.x & 31) / G * G));
    } else if constexpr (G >= kThreads) {
        __syncthreads();
    } else {
        if (g == X) asm volatile("bar.sync %0, %1;" ::"n"(X + 1), "n"(G) : "memory");
        else if constexpr (X + 1 < kThreads / G) group_sync<G, X + 1>(g);
    }
}

// The barrier of a box's step: a box's stages and metadata belong to its thread
// group, so whole warps meet their group only (256^3, FP64 half-sweep: 73.9 ->
// 72.2 us, FP32 restriction 50.7 -> 49.1 us); smaller groups meet the block.
// Returns whether to take the extra step: `extra` of this group's box, or of any
// box of the block.
template <int G>
__device__ __forceinline__ bool box_sync(int g, bool extra) {
    if constexpr (G >= 32) {
        group_sync<G>(g);
        return extra;
    } else {
        return __syncthreads_or(extra);
    }
}

// ---------------------------------------------------------------------------
// FP64 images in fixed point.  GB300 issues one FP64 instruction per 64 cycles
// and warp, and aligning every term of every sum to its cell's largest
// exponent (fx_sum) takes some 25 integer instructions a term.  A staged
// image is read seven times over, so it is aligned once instead: every value
// to the largest exponent E of the box and its ghosts, in place, as a 64-bit
// integer with G guard bits below the last bit of a value of that exponent
// (G = FxAcc<W>::G for sums of weight W: 7 for the half-sweep, 6 for the
// operator, 4 for the restriction in 3D).  Sums of neighbours are then integer
// additions, exact, rounded once.
//
// A box is aligned only where that loses no bit of any value (fx_common_exponent).
// So the aligned sums are the correctly rounded ones, and never further from the
// exact sum than the sums per cell (fx_sum, or FP64 additions), which a box of a
// wider span takes, and one whose largest exponent is out of fx_sum's range (all
// zero, infinite, NaN).  Where the sign of the field changes a box has small
// values beside large ones; such boxes are few (18.8 M unknowns, FP64: 21.5 ms
// with boxes of a span of 2^8 and more aligned too, 21.7 ms; 4.3 M, FP64, forward
// and adjoint, 24.3 and 24.8 ms).
// ---------------------------------------------------------------------------
template <int D>
constexpr int fx_lap_weight() { return 4 * D; }  // sum_nb u - 2D u

// A thread aligns what it staged itself, so finding E costs no pass over the
// image and no barrier of its own: after its wait a thread folds its values'
// magnitudes (fx_fold, every value by itself), its warp leaves their extremes in
// `red` (one int2 per warp, accessed as such: the type gives the array its 8-byte
// alignment) ahead of the barrier that every box has, every thread then knows E
// (fx_exponent), and after the alignment the group meets once more.
__device__ __forceinline__ void fx_leave(unsigned mx, unsigned mn, int2 *red) {
    mx = __reduce_max_sync(0xffffffffu, mx);
    mn = __reduce_min_sync(0xffffffffu, mn);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_int2((int)mx, (int)mn);
}
// exponent of group g's values, or -1 where they are not aligned (W: the sums' weight)
template <int G, int W>
__device__ __forceinline__ int fx_exponent(const int2 *red, int g) {
    static_assert(G >= 32, "whole warps per box");
    unsigned mx = 0, mn = 0xffffffffu;
#pragma unroll
    for (int x = 0; x < G / 32; ++x) {
        const int2 r = red[g * (G / 32) + x];
        mx = max(mx, (unsigned)r.x);
        mn = min(mn, (unsigned)r.y);
    }
    return fx_common_exponent<W>(mx, mn);
}
template <int W>
__device__ __forceinline__ void fx_align_at(double *p, int E, bool scalar) {
    if (scalar) {
        *p = __longlong_as_double(fx_align<W>(*p, E));
    } else {
        const double2 q = *reinterpret_cast<const double2 *>(p);
        *reinterpret_cast<longlong2 *>(p) = make_longlong2(fx_align<W>(q.x, E), fx_align<W>(q.y, E));
    }
}
// f(slot, scalar) for every value the thread staged through its plan
template <typename Plan, typename F>
__device__ __forceinline__ void fx_own(const Plan &pl, F f) {
#pragma unroll
    for (int it = 0; it < (int)(sizeof(pl.vdst) / sizeof(int)); ++it)
        if (pl.vdst[it] >= 0) f(pl.vdst[it], false);
#pragma unroll
    for (int q = 0; q < Plan::NQ; ++q)
        if (pl.gdst[q] >= 0) f(pl.gdst[q] & 0xffff, (pl.gdst[q] & (1 << 19)) != 0);
}
template <typename Plan>
__device__ __forceinline__ void fx_fold_own(const Plan &pl, const double *st, int2 *red) {
    unsigned mx = 0, mn = 0xffffffffu;
    fx_own(pl, [&](int q, bool scalar) {
        fx_fold(st[q], mx, mn);
        if (!scalar) fx_fold(st[q + 1], mx, mn);
    });
    fx_leave(mx, mn, red);
}

// resident blocks per SM the register allocation must allow (FP32 / FP64)
constexpr int kSmoothMinBlocks32 = 6, kSmoothMinBlocks64 = 5;

// The walk of a half-sweep: boxes staged through the ring, then per 16-byte
// vector of colour-c cells upd(I, v, itv, xl, xr, ym, yp, zm, zp, rv, out) forms
// the new values from the neighbours (in the order -x, +x, -y, +y, -z, +z) and
// the staged source.  early(I, v, itv) runs for the same vectors before the
// box's copies are waited for (loads of its own that upd needs).
// FX > 0 (FP64): the staged values are aligned (fx_align_at, sums of weight FX) and
// upd_fx(E, ...) forms the new values from them, upd only where they are not.
template <int D, int M, typename T, int VPT, int FX = 0, typename Early, typename Upd, typename UpdFx>
__device__ __forceinline__ void sp_walk(const BoxMeta &A, int b0, int n, const int *list, T *u,
                                        const T *__restrict__ rho, int colour, int hom, Early early, Upd upd,
                                        UpdFx upd_fx) {
    using S = SpCfg<D, M, T, VPT>;
    constexpr int VEC = S::VEC, MH = S::MH, H = S::H, NST = S::NST, NI = NST + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int g = threadIdx.x / S::G, lt = threadIdx.x % S::G;
    T *stages = reinterpret_cast<T *>(smem_raw);
    BoxInfo *info = reinterpret_cast<BoxInfo *>(smem_raw + sizeof(T) * S::BOX * S::BPC * NST);
    const int c = colour;
    const int stride = gridDim.x * S::BPC;
    const int first = blockIdx.x * S::BPC;
    SpPlan<D, M, T, VPT> pl;
    pl.init(lt, c);
    // per vector of this thread, the same for every box: the stage offset of
    // the x neighbour past the vector (half-row or x ghost) and the parity of
    // its row (the vector's own half-row is at pl.vdst)
    int cxoff[S::NIT];
    bool cr[S::NIT];
#pragma unroll
    for (int itv = 0; itv < S::NIT; ++itv) {
        const int v = lt + itv * S::G;
        const int row = v / S::NVR, h0 = (v % S::NVR) * VEC;
        const int j = row % M, k = D == 2 ? 0 : row / M;
        const int r = (c + j + k + D) & 1;
        const int pr_row = sp_row<D, M>(j, k);
        if (r) cxoff[itv] = h0 + VEC < MH ? pr_row * MH + h0 + VEC : S::PT + S::ROWS + pr_row;
        else cxoff[itv] = h0 > 0 ? pr_row * MH + h0 - 1 : S::PT + pr_row;
        cr[itv] = r;
    }
    pdl_trigger();
    __shared__ int2 fxr[FX ? kThreads / 32 : 1];
    for (int q = 0; q < NST; ++q)  // static metadata: before the wait
        info_stage<D>(A, first + q * stride + g, n, b0, list, info[q * S::BPC + g], lt, S::G);
    cp_commit();
    pdl_wait();
    cp_wait<0>();
    __syncthreads();
    for (int q = 0; q < NST - 1; ++q) {
        const BoxInfo &In = info[q * S::BPC + g];
        if (info_on(A, In)) sp_issue<D, M, T, VPT>(pl, In, u, rho, stages + (q * S::BPC + g) * S::BOX, lt, c);
        cp_commit();
    }
    int it = 0;
    for (int base = first; base < n; base += stride, ++it) {
        const BoxInfo &I = info[(it % NI) * S::BPC + g];
        const int b = info_on(A, I) ? I.b : -1;
        if (b >= 0) {
#pragma unroll
            for (int itv = 0; itv < S::NIT; ++itv)
                if (lt + itv * S::G < S::NV) early(I, lt + itv * S::G, itv);
        }
        cp_wait<NST - 2>();  // this box's copies (issued NST-1 boxes ago) have landed
        const bool special = b >= 0 && (I.flag & BF_SPECIAL);
        const bool cf = b >= 0 && (I.flag & BF_CF);
        T *box = stages + ((it % NST) * S::BPC + g) * S::BOX;
        if (special) sp_fix_own<D, M, T, VPT>(pl, I, A, box, hom);  // domain sides: this thread's own items
        if constexpr (FX > 0) {
            if (b >= 0) fx_fold_own(pl, box, fxr);
        }
        // one barrier per box: the stage and metadata slot of the previous box are free after it
        const int any_cf = box_sync<S::G>(g, cf);
        {
            const int q = it + NST - 1;
            const BoxInfo &In = info[(q % NI) * S::BPC + g];
            if (info_on(A, In))
                sp_issue<D, M, T, VPT>(pl, In, u, rho, stages + ((q % NST) * S::BPC + g) * S::BOX, lt, c);
            info_stage<D>(A, base + NST * stride + g, n, b0, list, info[((it + NST) % NI) * S::BPC + g], lt, S::G);
            cp_commit();
        }
        if (any_cf) {  // refinement-boundary ghosts read cells other threads staged
            if (cf) {
                sp_fix<D, M, T, VPT>(I, A, u, box, lt, c, hom, true);
                if constexpr (FX > 0) fx_fold_own(pl, box, fxr);  // the thread's own items again
            }
            box_sync<S::G>(g, false);
        }
        if (b >= 0) {
            const T *R = box + S::PT + S::XT;
            auto cells = [&](auto form) {
#pragma unroll
            for (int itv = 0; itv < S::NIT; ++itv) {
                if (lt + itv * S::G >= S::NV) continue;
                const T *pr = box + pl.vdst[itv];  // the vector's colour 1-c half-row
                T xv[VEC], ym[VEC], yp[VEC], zm[VEC], zp[VEC], rv[VEC];
                ldv<T, VEC>(pr, xv);
                const T extra = box[cxoff[itv]];
                ldv<T, VEC>(pr - MH, ym);
                ldv<T, VEC>(pr + MH, yp);
                if (D == 3) {
                    ldv<T, VEC>(pr - (M + 2) * MH, zm);
                    ldv<T, VEC>(pr + (M + 2) * MH, zp);
                }
                ldv<T, VEC>(R + (lt + itv * S::G) * VEC, rv);
                const bool r = cr[itv];
                // the x neighbours: the cell's own half-row entry and the one beside it
                // (towards +x for r = 1, towards -x for r = 0; `extra` past the vector)
                T xl[VEC], xr[VEC], out[VEC];
#pragma unroll
                for (int x = 0; x < VEC; ++x) {
                    const T side = r ? (x + 1 < VEC ? xv[x + 1] : extra) : (x ? xv[x - 1] : extra);
                    xl[x] = r ? xv[x] : side;
                    xr[x] = r ? side : xv[x];
                }
                form(I, lt + itv * S::G, itv, xl, xr, ym, yp, zm, zp, rv, out);
                stv<T, VEC>(u + I.coff + c * H + (lt + itv * S::G) * VEC, out);
            }
            };
            if constexpr (FX > 0) {
                const int E = fx_exponent<S::G, FX>(fxr, g);
                if (E >= 0) fx_own(pl, [&](int q, bool scalar) { fx_align_at<FX>(box + q, E, scalar); });
                group_sync<S::G>(g);
                if (E >= 0)
                    cells([&](const BoxInfo &, int, int, const T (&xl)[VEC], const T (&xr)[VEC], const T (&ym)[VEC],
                              const T (&yp)[VEC], const T (&zm)[VEC], const T (&zp)[VEC], const T (&rv)[VEC],
                              T (&out)[VEC]) { upd_fx(E, xl, xr, ym, yp, zm, zp, rv, out); });
                else cells(upd);
            } else {
                cells(upd);
            }
        }
    }
    cp_wait<0>();
}

// FP64 half-sweeps in 3D whose boxes take whole warps align their images: 256^3
// 100.5 -> 72.2 us, 201 instead of 249 instructions and one instead of five FP64
// issues per update; 18.8 M unknowns, FP64, 29.0 -> 23.3 ms with the restriction
// and the coarse right-hand side on aligned images too (2D keeps the per-cell
// sums: its four terms need no FP64 addition).  With info_stage 66 us: issue
// bound, 52.7 M warp instructions and 191 MB of DRAM traffic (2.9 TB/s) a launch.
template <int D, int M, typename T, int VPT>
constexpr bool fx_smooth() { return sizeof(T) == 8 && D == 3 && SpCfg<D, M, T, VPT>::G >= 32; }

// FP64: rho holds -h^2 rho / (2D) and the update is u = sum/(2D) + rho (a choice
// at run time would cost the other form's two FP64 instructions per update,
// which the compiler runs too and selects)
template <int D, int M, typename T, int VPT = 1>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? kSmoothMinBlocks32 : kSmoothMinBlocks64)
    k_smooth_p(BoxMeta A, int b0, int n, const int *list, T *u, const T *__restrict__ rho, T h2, int colour, int hom) {
    constexpr int VEC = SpCfg<D, M, T, VPT>::VEC;
    constexpr bool kScaled = sizeof(T) == 8;
    const T inv = T(1) / T(2 * D);
    auto early = [](const BoxInfo &, int, int) {};
    auto upd = [&](const BoxInfo &, int, int, const T (&xl)[VEC], const T (&xr)[VEC], const T (&ym)[VEC],
                   const T (&yp)[VEC], const T (&zm)[VEC], const T (&zp)[VEC], const T (&rv)[VEC], T (&out)[VEC]) {
#pragma unroll
        for (int x = 0; x < VEC; ++x) {
            const T sum = nb_sum6<D, T>(xl[x], xr[x], ym[x], yp[x], D == 3 ? zm[x] : T(0), D == 3 ? zp[x] : T(0));
            out[x] = kScaled ? fma(sum, inv, rv[x]) : (sum - h2 * rv[x]) * inv;
        }
    };
    auto upd_fx = [&](int E, const T (&xl)[VEC], const T (&xr)[VEC], const T (&ym)[VEC], const T (&yp)[VEC],
                      const T (&zm)[VEC], const T (&zp)[VEC], const T (&rv)[VEC], T (&out)[VEC]) {
        auto i = [](T v) { return __double_as_longlong(v); };
#pragma unroll
        for (int x = 0; x < VEC; ++x) {
            const long long S = i(xl[x]) + i(xr[x]) + i(ym[x]) + i(yp[x]) + i(zm[x]) + i(zp[x]);
            out[x] = fma(fx_round<2 * D>(S, E), inv, rv[x]);
        }
    };
    constexpr int FX = fx_smooth<D, M, T, VPT>() ? 2 * D : 0;
    sp_walk<D, M, T, VPT, FX>(A, b0, n, list, u, rho, colour, hom, early, upd, upd_fx);
}

}  // namespace afg
