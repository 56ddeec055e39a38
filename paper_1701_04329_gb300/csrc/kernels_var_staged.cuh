// Variable-coefficient operators (arXiv:1701.04329 Sec. 3.4-3.5) with stored
// face coefficients: the staged kernels of the Laplacian (kernels_smooth.cuh,
// kernels_full.cuh) with a coefficient per face.
//
// The coefficients of a cell's 2D faces (the harmonic means of eps, in (r,z)
// weighted by r_face / r_cell) do not change while eps stands, but forming
// them takes a division per face: in FP64 some 14 instructions of a unit
// that issues one per 64 cycles and warp, which was nine tenths of a half-sweep
// (kernels_var.cuh), and in FP32 most of its instructions.  They are formed
// once per eps and level (k_var_coef) and kept, per cell, as 2D + 2 arrays in
// the box layout:
//   c_0 .. c_{2D-1}  the face coefficients, order -x, +x, -y, +y, -z, +z
//   s                their sum in that order
//   1/s
// A half-sweep reads each of them once, as 16-byte vectors straight into
// registers (no other cell uses them), issued before the wait for the box's
// staged values.  The local solve (sum_s c_s u_s - h^2 rho) / s is the
// quotient q = n (1/s) corrected by its exact remainder, q + (n - q s)(1/s):
// the rounding of a division without its chain.
//
// Measured on a GB300: a solve of 107 k unknowns in 2D, FP64, 14.0 -> 6.6 ms;
// 3.5 M unknowns in 3D, mixed, 16.9 -> 8.0 ms; 294 k unknowns in (r,z), mixed,
// 8.2 -> 5.8 ms; the same solutions bit for bit.
#pragma once
#include "kernels_full.cuh"
#include "kernels_var.cuh"
#include "var_ops.cuh"

namespace afg {

// c: first coefficient array; the arrays follow each other, n values apart
template <typename T>
struct VarCoef {
    const T *c;
    long long n;
};

template <int D, int M, typename T>
__global__ void __launch_bounds__(kThreads) k_var_coef(BoxMeta A, int b0, int n, const T *eps, T *out, long long nc,
                                                       int op) {
    using S = VarCfg<D, M, T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int g = threadIdx.x / S::G, lt = threadIdx.x % S::G;
    T *E = reinterpret_cast<T *>(smem_raw) + g * S::BOX;
    BoxInfo *info;
    short *tix, *gt, *gs;
    carve<D, M>(smem_raw, sizeof(T) * S::BOX * S::BPC, S::BPC, info, tix, gt, gs);
    pdl_trigger();
    build_tables<D, M>(tix, gt, gs, -1);
    pdl_wait();
    for (int base = blockIdx.x * S::BPC; base < n; base += gridDim.x * S::BPC) {
        __syncthreads();
        info_load<D>(A, base + g, n, b0, nullptr, info[g], lt, S::G, false);
        __syncthreads();
        const BoxInfo &I = info[g];
        if (I.b >= 0) gather_eps<D, M, T, S::G>(I, eps, E, lt, tix, gt, gs);
        __syncthreads();
        if (I.b < 0) continue;
        const T h = T(A.hb[I.b]), x0 = T(A.x0[I.b]);
        for (int q = lt; q < S::C; q += S::G) {
            int i, j, k;
            rb_cell<D, M>(q, i, j, k);
            T c[2 * D], s = T(0);
            var_coef<D, M, T>(E, tix[q], i, h, x0, op, c);
#pragma unroll
            for (int f = 0; f < 2 * D; ++f) {
                out[f * nc + I.coff + q] = c[f];
                s += c[f];
            }
            out[2 * D * nc + I.coff + q] = s;
            out[(2 * D + 1) * nc + I.coff + q] = T(1) / s;
        }
    }
}

// Half-sweep: per update 2D + 2 FMAs and a multiplication instead of 2D
// divisions; 2D + 2 coefficient values read per updated cell.
template <int D, int M, typename T>
__global__ void __launch_bounds__(kThreads) k_var_smooth_p(BoxMeta A, int b0, int n, T *u, const T *__restrict__ rho,
                                                           VarCoef<T> V, T h2, int colour, int hom) {
    using S = SpCfg<D, M, T>;
    constexpr int VEC = S::VEC, NC = 2 * D + 2;
    T cf[S::NIT][NC][VEC];
    auto early = [&](const BoxInfo &I, int v, int itv) {
        const T *p = V.c + I.coff + colour * S::H + v * VEC;
#pragma unroll
        for (int f = 0; f < NC; ++f) ldv<T, VEC>(p + f * V.n, cf[itv][f]);
    };
    auto upd = [&](const BoxInfo &, int, int itv, const T (&xl)[VEC], const T (&xr)[VEC], const T (&ym)[VEC],
                   const T (&yp)[VEC], const T (&zm)[VEC], const T (&zp)[VEC], const T (&rv)[VEC], T (&out)[VEC]) {
#pragma unroll
        for (int x = 0; x < VEC; ++x) {
            T c[2 * D], w[2 * D];
#pragma unroll
            for (int s = 0; s < 2 * D; ++s) c[s] = cf[itv][s][x];
            w[0] = xl[x]; w[1] = xr[x]; w[2] = ym[x]; w[3] = yp[x];
            if constexpr (D == 3) { w[4] = zm[x]; w[5] = zp[x]; }
            out[x] = var_quot<T>(fma(-h2, rv[x], var_dot<D, T>(c, w)), cf[itv][2 * D][x], cf[itv][2 * D + 1][x]);
        }
    };
    sp_walk<D, M, T, 1>(A, b0, n, nullptr, u, rho, colour, hom, early, upd, [](auto &&...) {});
}

// For the VEC cells of colour col at half-row (j,k), h0..h0+VEC-1 (storage
// position q0): sum_s c_s u_s - (sum_s c_s) u, h^2 times the operator.
template <int D, int M, typename T>
__device__ __forceinline__ void fp_var_lap_vec(const T *st, const T *cp, long long nc, int col, int j, int k, int h0,
                                               T *lap, T *self) {
    using F = FpCfg<D, M, T>;
    constexpr int VEC = F::VEC, MH = F::MH;
    T cf[2 * D + 1][VEC];
#pragma unroll
    for (int f = 0; f <= 2 * D; ++f) ldv<T, VEC>(cp + f * nc, cf[f]);
    const int rowi = sp_row<D, M>(j, k);
    const int r = (col + j + k + D) & 1;
    const T *po = st + (1 - col) * F::PT + rowi * MH + h0;
    const T *X = st + 2 * F::PT;
    T xv[VEC], ym[VEC], yp[VEC], zm[VEC], zp[VEC];
    ldv<T, VEC>(st + col * F::PT + rowi * MH + h0, self);
    ldv<T, VEC>(po, xv);
    T extra;
    if (r) extra = h0 + VEC < MH ? po[VEC] : X[F::ROWS + rowi];
    else extra = h0 > 0 ? po[-1] : X[rowi];
    ldv<T, VEC>(po - MH, ym);
    ldv<T, VEC>(po + MH, yp);
    if (D == 3) {
        ldv<T, VEC>(po - (M + 2) * MH, zm);
        ldv<T, VEC>(po + (M + 2) * MH, zp);
    }
#pragma unroll
    for (int x = 0; x < VEC; ++x) {
        T c[2 * D], w[2 * D];
#pragma unroll
        for (int s = 0; s < 2 * D; ++s) c[s] = cf[s][x];
        w[0] = r ? xv[x] : (x ? xv[x - 1] : extra);
        w[1] = r ? (x + 1 < VEC ? xv[x + 1] : extra) : xv[x];
        w[2] = ym[x]; w[3] = yp[x];
        if constexpr (D == 3) { w[4] = zm[x]; w[5] = zp[x]; }
        lap[x] = fma(-cf[2 * D][x], self[x], var_dot<D, T>(c, w));
    }
}

// Residual and restriction: the residual of every cell replaces its source in
// the stage, then the mean of the 2^D children (weighted by r in (r,z)) goes
// to the parent.
template <int D, int M, int MP, typename T>
__global__ void __launch_bounds__(kThreads) k_var_resid_restrict_p(BoxMeta A, int b0, int n, T *u, T *rho, T *vold,
                                                                   VarCoef<T> V, T ih2, int hom, int op) {
    constexpr int GT = fas_threads<D, M, T>();
    using F = FpCfg<D, M, T, GT>;
    constexpr int MH = M / 2, VEC = F::VEC, NVH = F::H / VEC;
    constexpr int NCO = D == 2 ? MH * MH : MH * MH * MH;
    pdl_trigger();
    auto want = [](const BoxInfo &) { return true; };
    auto flat = [&](const BoxInfo &) -> const T * { return rho; };
    auto body = [&](const BoxInfo &I, T *st, int lt, int) {
        T *R = st + F::UB;
        for (int v = lt; v < F::NV; v += F::G) {
            const int col = v / NVH, w = v % NVH;
            const int row = w / F::NVR, h0 = (w % F::NVR) * VEC;
            const int j = row % M, k = D == 2 ? 0 : row / M;
            T lap[VEC], self[VEC], rv[VEC];
            fp_var_lap_vec<D, M, T>(st, V.c + I.coff + v * VEC, V.n, col, j, k, h0, lap, self);
            ldv<T, VEC>(R + v * VEC, rv);
#pragma unroll
            for (int x = 0; x < VEC; ++x) rv[x] = fma(-lap[x], ih2, rv[x]);
            stv<T, VEC>(R + v * VEC, rv);
        }
        group_sync<GT>(threadIdx.x / GT);
        const long long cp = A.coff[I.parent];
        const T h = T(A.hb[I.b]), x0 = T(A.x0[I.b]);
        for (int c = lt; c < NCO; c += F::G) {
            const int X = c % MH, Y = (c / MH) % MH, Z = D == 3 ? c / (MH * MH) : 0;
            T su = T(0), sr = T(0), sw = T(0);
#pragma unroll
            for (int dz = 0; dz < (D == 3 ? 2 : 1); ++dz)
#pragma unroll
                for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                    for (int dx = 0; dx < 2; ++dx) {
                        const int i = 2 * X + dx, j = 2 * Y + dy, k = D == 3 ? 2 * Z + dz : 0;
                        const T uu = st[fp_slot<D, M, T>(i, j, k)], rr = R[rbi<D, M>(i, j, k)];
                        if (op == 2) {
                            const T w = var_weight<T>(op, x0, h, i);
                            su += w * uu;
                            sr += w * rr;
                            sw += w;
                        } else {
                            su += uu;
                            sr += rr;
                        }
                    }
            const int pi = unpack_off(I.poff, 0) + X, pj = unpack_off(I.poff, 1) + Y;
            const int pk = D == 3 ? unpack_off(I.poff, 2) + Z : 0;
            const long long q = cp + rbi<D, MP>(pi, pj, pk);
            const T w = T(1) / T(1 << D);
            const T mu = op == 2 ? su / sw : su * w;
            u[q] = mu;
            vold[q] = mu;
            rho[q] = op == 2 ? sr / sw : sr * w;
        }
    };
    auto none = [](const BoxInfo *) {};
    fp_walk<D, M, T, GT>(A, b0, n, nullptr, u, hom, want, flat, body, none, none);
}

// FAS coarse right-hand side: refined boxes rho_H += A_H(v_H), leaves v' = v.
template <int D, int M, typename T>
__global__ void __launch_bounds__(kThreads) k_var_fas_p(BoxMeta A, int b0, int n, const T *u, T *rho, T *vold,
                                                        VarCoef<T> V, T ih2, int hom) {
    constexpr int GT = fas_threads<D, M, T>();
    using F = FpCfg<D, M, T, GT>;
    constexpr int VEC = F::VEC, NVH = F::H / VEC;
    pdl_trigger();
    auto want = [](const BoxInfo &I) { return (I.flag & BF_REFINED) != 0; };
    auto flat = [&](const BoxInfo &I) -> const T * { return (I.flag & BF_REFINED) ? rho : u; };
    auto body = [&](const BoxInfo &I, const T *st, int lt, int) {
        const T *FL = st + F::UB;
        for (int v = lt; v < F::NV; v += F::G) {
            T rv[VEC];
            ldv<T, VEC>(FL + v * VEC, rv);
            if (!(I.flag & BF_REFINED)) {
                stv<T, VEC>(vold + I.coff + (long long)v * VEC, rv);
                continue;
            }
            const int col = v / NVH, w = v % NVH;
            const int row = w / F::NVR, h0 = (w % F::NVR) * VEC;
            const int j = row % M, k = D == 2 ? 0 : row / M;
            T lap[VEC], self[VEC];
            fp_var_lap_vec<D, M, T>(st, V.c + I.coff + v * VEC, V.n, col, j, k, h0, lap, self);
#pragma unroll
            for (int x = 0; x < VEC; ++x) rv[x] = fma(lap[x], ih2, rv[x]);
            stv<T, VEC>(rho + I.coff + (long long)v * VEC, rv);
        }
    };
    auto none = [](const BoxInfo *) {};
    fp_walk<D, M, T, GT>(A, b0, n, nullptr, u, hom, want, flat, body, none, none);
}

// Composite residual on the leaves with its norms per tree, and r in rout.
template <int D, int M, typename T, typename R, bool ONE>
__global__ void __launch_bounds__(kThreads) k_var_leaf_residual_p(BoxMeta A, const int *list, int n, const T *u,
                                                                  const T *__restrict__ rho, VarCoef<T> V, int hom,
                                                                  unsigned long long *rmax, unsigned long long *pmax,
                                                                  R *rout) {
    constexpr int GT = leaf_threads<D, M, T, R>();
    constexpr int VEC = FpCfg<D, M, T, GT>::VEC;
    pdl_trigger();
    auto lap = [&](const BoxInfo &I, const T *st, int v, int col, int j, int k, int h0, T *out) {
        T self[VEC];
        fp_var_lap_vec<D, M, T>(st, V.c + I.coff + v * VEC, V.n, col, j, k, h0, out, self);
    };
    leaf_residual_walk<D, M, T, R, GT, 0, ONE>(A, list, n, u, rho, hom, rmax, pmax, rout, lap);
}

}  // namespace afg
