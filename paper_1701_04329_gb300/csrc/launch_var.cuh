// Launches of the variable-coefficient kernels (kernels_var.cuh), included
// by launch_var_d2.cu / launch_var_d3.cu (one translation unit per
// dimension, compiled in parallel).
#pragma once
#include "kernels_prolong.cuh"
#include "kernels_transfer.cuh"
#include "kernels_var_staged.cuh"
#include "launch_impl.cuh"

namespace afg {

// The staged kernels with stored coefficients wherever a half-row holds a
// 16-byte vector; the others (grids of 2 cells per side, and of 4 in FP32), and
// all grids where the coefficients are not kept (W.coef null), take the kernels
// that form the coefficients from eps.
template <int D, int M, typename T>
void do_var_coef(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *eps, void *coef, long long nc,
                 int op) {
    if (n <= 0) return;
    using S = VarCfg<D, M, T>;
    auto k = k_var_coef<D, M, T>;
    launch_pdl(k, grid_for(k, S::smem(), (n + S::BPC - 1) / S::BPC), S::smem(), c.stream, A, b0, n, (const T *)eps,
               (T *)coef, nc, op);
    ++g_launches;
}

template <int D, int M, typename T>
void do_var_smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *rho, const VarArgs &W,
                   int colour, int hom) {
    if (n <= 0) return;
    if constexpr (SpCfg<D, M, T>::ok) {
        if (W.coef) {
            using S = SpCfg<D, M, T>;
            auto k = k_var_smooth_p<D, M, T>;
            const VarCoef<T> V{(const T *)W.coef, W.n};
            launch_pdl(k, grid_for(k, S::smem(), (n + S::BPC - 1) / S::BPC), S::smem(), c.stream, A, b0, n, (T *)u,
                       (const T *)rho, V, T(W.h * W.h), colour, hom);
            ++g_launches;
            return;
        }
    }
    const void *eps = W.eps;
    const int op = W.op;
    using S = VarCfg<D, M, T>;
    auto k = k_var_smooth<D, M, T>;
    launch_pdl(k, grid_for(k, S::smem(), (n + S::BPC - 1) / S::BPC), S::smem(), c.stream, A, b0, n, (T *)u,
               (const T *)rho, (const T *)eps, colour, hom, op);
    ++g_launches;
}

template <int D, int M, int MP, typename T>
void do_var_resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                           const VarArgs &W, int hom) {
    if (n <= 0) return;
    if constexpr (FpCfg<D, M, T>::ok) {
        if (W.coef) {
            using F = FpCfg<D, M, T, fas_threads<D, M, T>()>;
            auto k = k_var_resid_restrict_p<D, M, MP, T>;
            const VarCoef<T> V{(const T *)W.coef, W.n};
            launch_pdl(k, grid_for(k, F::smem(), (n + F::BPC - 1) / F::BPC), F::smem(), c.stream, A, b0, n, (T *)u,
                       (T *)rho, (T *)vold, V, T(1.0 / (W.h * W.h)), hom, W.op);
            ++g_launches;
            return;
        }
    }
    const void *eps = W.eps;
    const int op = W.op;
    using S = VarCfg<D, M, T>;
    auto k = k_var_resid_restrict<D, M, MP, T>;
    launch_pdl(k, grid_for(k, S::smem(), (n + S::BPC - 1) / S::BPC), S::smem(), c.stream, A, b0, n, (T *)u, (T *)rho,
               (T *)vold, (const T *)eps, hom, op);
    ++g_launches;
}

template <int D, int M, typename T>
void do_var_fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold,
                const VarArgs &W, int hom) {
    if (n <= 0) return;
    if constexpr (FpCfg<D, M, T>::ok) {
        if (W.coef) {
            using F = FpCfg<D, M, T, fas_threads<D, M, T>()>;
            auto k = k_var_fas_p<D, M, T>;
            const VarCoef<T> V{(const T *)W.coef, W.n};
            launch_pdl(k, grid_for(k, F::smem(), (n + F::BPC - 1) / F::BPC), F::smem(), c.stream, A, b0, n, (const T *)u,
                       (T *)rho, (T *)vold, V, T(1.0 / (W.h * W.h)), hom);
            ++g_launches;
            return;
        }
    }
    const void *eps = W.eps;
    const int op = W.op;
    using S = VarCfg<D, M, T>;
    auto k = k_var_fas<D, M, T>;
    launch_pdl(k, grid_for(k, S::smem(), (n + S::BPC - 1) / S::BPC), S::smem(), c.stream, A, b0, n, (const T *)u,
               (T *)rho, (T *)vold, (const T *)eps, hom, op);
    ++g_launches;
}

template <int D, int M, typename T, typename Ro>
void do_var_leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,
                          const void *rho, const VarArgs &W, int hom, unsigned long long *rmax,
                          unsigned long long *pmax, void *rout) {
    if (n <= 0) return;
    static_assert(FpCfg<D, M, T>::ok, "leaf boxes have 4 cells per side or more, in FP64");
    if (W.coef) {
        using F = FpCfg<D, M, T, leaf_threads<D, M, T, Ro>()>;
        auto k = c.one_tree ? k_var_leaf_residual_p<D, M, T, Ro, true> : k_var_leaf_residual_p<D, M, T, Ro, false>;
        const VarCoef<T> V{(const T *)W.coef, W.n};
        launch_pdl(k, grid_for(k, F::smem(), (n + F::BPC - 1) / F::BPC), F::smem(), c.stream, A, list, n,
                   (const T *)u, (const T *)rho, V, hom, rmax, pmax, (Ro *)rout);
    } else {
        using S = VarCfg<D, M, T>;
        auto k = k_var_leaf_residual<D, M, T, Ro>;
        launch_pdl(k, grid_for(k, S::smem(), (n + S::BPC - 1) / S::BPC), S::smem(), c.stream, A, list, n,
                   (const T *)u, (const T *)rho, (const T *)W.eps, hom, W.op, rmax, pmax, (Ro *)rout);
    }
    ++g_launches;
}

template <int D, int M, int MP, typename T>
void do_var_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *v, int op) {
    if (n <= 0) return;
    constexpr int NCO = D == 2 ? (M / 2) * (M / 2) : (M / 2) * (M / 2) * (M / 2);
    auto k = k_var_restrict<D, M, MP, T>;
    const long long work = ((long long)n * NCO + kThreads - 1) / kThreads;
    launch_pdl(k, grid_for(k, 0, (int)std::min<long long>(work, 1 << 20)), 0, c.stream, A, b0, n, list, (T *)v, op);
    ++g_launches;
}

template <int D, int M, int MP, typename T>
void do_correct_x(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold, const int *nball,
                  int scheme) {
    if (n <= 0) return;
    using S = PxCfg<D, M>;
    const size_t smem = S::template smem<T>();
    auto k = k_correct_x<D, M, MP, T>;
    launch_pdl(k, grid_for(k, smem, (n + S::BPC - 1) / S::BPC), smem, c.stream, A, b0, n, (T *)u, (const T *)vold,
               nball, scheme);
    ++g_launches;
}

template <int D, int M>
void do_transfer(cudaStream_t st, const BoxMeta &Ao, const double *uo, const int *nball_o, const BoxMeta &An,
                 double *un, const int *new_leaves, const int *src, const int *poff, int n, int scheme) {
    if (n <= 0) return;
    using S = TrCfg<D, M>;
    const size_t smem = S::template smem<double>();
    auto k = k_transfer<D, M, double>;
    launch_pdl(k, grid_for(k, smem, (n + S::BPC - 1) / S::BPC), smem, st, Ao, uo, nball_o, An, un, new_leaves, src,
               poff, n, scheme);
    ++g_launches;
}

template <int D>
struct VarOps {
    static void transfer(cudaStream_t st, int N, const BoxMeta &Ao, const double *uo, const int *nball_o,
                         const BoxMeta &An, double *un, const int *new_leaves, const int *src, const int *poff, int n,
                         int scheme) {
        switch (N) {
            case 4: do_transfer<D, 4>(st, Ao, uo, nball_o, An, un, new_leaves, src, poff, n, scheme); break;
            case 8: do_transfer<D, 8>(st, Ao, uo, nball_o, An, un, new_leaves, src, poff, n, scheme); break;
            case 16: do_transfer<D, 16>(st, Ao, uo, nball_o, An, un, new_leaves, src, poff, n, scheme); break;
            default: bad_size(N, 0);
        }
    }
    template <typename T>
    static void correct_x(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold,
                          const int *nball, int scheme) {
        AFG_SWITCH_MMP(c.M, c.MP, (do_correct_x<D, MM, PP, T>(c, A, b0, n, u, vold, nball, scheme)));
    }
    template <typename T>
    static void coef(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *eps, void *out, long long nc,
                     int op) {
        AFG_SWITCH_M(c.M, (do_var_coef<D, MM, T>(c, A, b0, n, eps, out, nc, op)));
    }
    template <typename T>
    static void smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *rho, const VarArgs &W,
                       int colour, int hom) {
        AFG_SWITCH_M(c.M, (do_var_smooth<D, MM, T>(c, A, b0, n, u, rho, W, colour, hom)));
    }
    template <typename T>
    static void resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                               const VarArgs &W, int hom) {
        AFG_SWITCH_MMP(c.M, c.MP, (do_var_resid_restrict<D, MM, PP, T>(c, A, b0, n, u, rho, vold, W, hom)));
    }
    template <typename T>
    static void fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold,
                    const VarArgs &W, int hom) {
        AFG_SWITCH_M(c.M, (do_var_fas<D, MM, T>(c, A, b0, n, u, rho, vold, W, hom)));
    }
    template <typename T>
    static void restrict_v(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *v, int op) {
        AFG_SWITCH_MMP(c.M, c.MP, (do_var_restrict<D, MM, PP, T>(c, A, b0, n, list, v, op)));
    }
    static void leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,
                              const void *rho, const VarArgs &W, int hom, unsigned long long *rmax,
                              unsigned long long *pmax, void *rout, bool rout_f32) {
        switch (c.M) {
            case 4: go<4>(c, A, list, n, u, rho, W, hom, rmax, pmax, rout, rout_f32); break;
            case 8: go<8>(c, A, list, n, u, rho, W, hom, rmax, pmax, rout, rout_f32); break;
            case 16: go<16>(c, A, list, n, u, rho, W, hom, rmax, pmax, rout, rout_f32); break;
            default: bad_size(c.M, 0);
        }
    }
    template <int M>
    static void go(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u, const void *rho,
                   const VarArgs &W, int hom, unsigned long long *rmax, unsigned long long *pmax, void *rout,
                   bool rout_f32) {
        if (rout_f32) do_var_leaf_residual<D, M, double, float>(c, A, list, n, u, rho, W, hom, rmax, pmax, rout);
        else do_var_leaf_residual<D, M, double, double>(c, A, list, n, u, rho, W, hom, rmax, pmax, rout);
    }
};

// the entry points of launch.h for one dimension
#define AFG_VAR_LAUNCHES(DD)                                                                                          \
    void launch_var_coef_d##DD(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *eps, void *out,       \
                               long long nc, int op) {                                                                \
        if (c.fp64) VarOps<DD>::coef<double>(c, A, b0, n, eps, out, nc, op);                                          \
        else VarOps<DD>::coef<float>(c, A, b0, n, eps, out, nc, op);                                                  \
    }                                                                                                                 \
    void launch_var_smooth_d##DD(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *rho,       \
                                 const VarArgs &W, int colour, int hom) {                                             \
        if (c.fp64) VarOps<DD>::smooth<double>(c, A, b0, n, u, rho, W, colour, hom);                                  \
        else VarOps<DD>::smooth<float>(c, A, b0, n, u, rho, W, colour, hom);                                          \
    }                                                                                                                 \
    void launch_var_resid_restrict_d##DD(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho,     \
                                         void *vold, const VarArgs &W, int hom) {                                     \
        if (c.fp64) VarOps<DD>::resid_restrict<double>(c, A, b0, n, u, rho, vold, W, hom);                            \
        else VarOps<DD>::resid_restrict<float>(c, A, b0, n, u, rho, vold, W, hom);                                    \
    }                                                                                                                 \
    void launch_var_fas_d##DD(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho,          \
                              void *vold, const VarArgs &W, int hom) {                                                \
        if (c.fp64) VarOps<DD>::fas<double>(c, A, b0, n, u, rho, vold, W, hom);                                       \
        else VarOps<DD>::fas<float>(c, A, b0, n, u, rho, vold, W, hom);                                               \
    }                                                                                                                 \
    void launch_var_restrict_d##DD(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *v,     \
                                   int op) {                                                                          \
        if (c.fp64) VarOps<DD>::restrict_v<double>(c, A, b0, n, list, v, op);                                        \
        else VarOps<DD>::restrict_v<float>(c, A, b0, n, list, v, op);                                                 \
    }                                                                                                                 \
    void launch_correct_x_d##DD(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold,      \
                                const int *nball, int scheme) {                                                       \
        if (c.fp64) VarOps<DD>::correct_x<double>(c, A, b0, n, u, vold, nball, scheme);                               \
        else VarOps<DD>::correct_x<float>(c, A, b0, n, u, vold, nball, scheme);                                       \
    }                                                                                                                 \
    void launch_transfer_d##DD(cudaStream_t st, int N, const BoxMeta &Ao, const double *uo, const int *nball_o,      \
                               const BoxMeta &An, double *un, const int *new_leaves, const int *src,                  \
                               const int *poff, int n, int scheme) {                                                  \
        VarOps<DD>::transfer(st, N, Ao, uo, nball_o, An, un, new_leaves, src, poff, n, scheme);                       \
    }                                                                                                                 \
    void launch_var_leaf_residual_d##DD(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,  \
                                        const void *rho, const VarArgs &W, int hom, unsigned long long *rmax,         \
                                        unsigned long long *pmax, void *rout, bool rout_f32) {                        \
        VarOps<DD>::leaf_residual(c, A, list, n, u, rho, W, hom, rmax, pmax, rout, rout_f32);                         \
    }

}  // namespace afg
