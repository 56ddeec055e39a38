// Template side of the launch layer; instantiated per dimension (the
// dispatch, launch_d2.cu / launch_d3.cu) and per dimension and precision (the
// launches and their kernels, launch_d<D>_f64.cu / launch_d<D>_f32.cu), so
// that the six translation units compile in parallel.
#pragma once
#include <algorithm>
#include <stdexcept>
#include <string>

#include "kernels_leaf.cuh"
#include "kernels_smooth.cuh"
#include "kernels_full.cuh"
#include "kernels_coarse.cuh"
#include "launch.h"

namespace afg {

int sm_count();
// resident CTAs per SM of a kernel for a given dynamic shared memory size (cached)
int occupancy(const void *kernel, size_t smem);

// Persistent grid: (resident CTAs per SM) x SMs, capped by the work.
template <typename K>
int grid_for(K kernel, size_t smem, int work_ctas) {
    const int cap = occupancy(reinterpret_cast<const void *>(kernel), smem) * sm_count();
    return std::max(1, std::min(work_ctas, cap));
}

// Launch with programmatic stream serialization (PDL): the kernel may start
// while its predecessor drains; every kernel waits (griddepcontrol.wait)
// before reading data a predecessor wrote.
template <typename... KArgs, typename... Args>
void launch_pdl_block(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
void launch_pdl(void (*kernel)(KArgs...), int grid, size_t smem, cudaStream_t s, Args... args) {
    launch_pdl_block(kernel, grid, kThreads, smem, s, args...);
}

template <int D, int M>
inline int work_ctas(int nbox) { return (nbox + Geo<D, M>::BPC - 1) / Geo<D, M>::BPC; }

template <int D, int M, typename T>
void do_smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u, const void *rho,
               const void *rhoh, double h2, int colour, int hom) {
    if (n <= 0) return;
    // the staged half-row kernel wherever a half-row holds a 16-byte vector
    if constexpr (SpCfg<D, M, T>::ok) {
        // FP32 with half the threads per box (two vectors per thread) on request
        if constexpr (sizeof(T) == 4 && SpCfg<D, M, T>::NV >= 2) {
            if (c.vpt == 2) {
                using S = SpCfg<D, M, T, 2>;
                const size_t smem = S::smem();
                auto k = k_smooth_p<D, M, T, 2>;
                launch_pdl(k, grid_for(k, smem, (n + S::BPC - 1) / S::BPC), smem, c.stream, A, b0, n, list, (T *)u,
                           (const T *)rho, T(h2), colour, hom);
                ++g_launches;
                return;
            }
        }
        {
            using S = SpCfg<D, M, T>;
            const size_t smem = S::smem();
            auto k = k_smooth_p<D, M, T>;
            if (sizeof(T) == 8 && !rhoh) throw std::runtime_error("FP64 half-sweeps read the pre-scaled source");
            launch_pdl(k, grid_for(k, smem, (n + S::BPC - 1) / S::BPC), smem, c.stream, A, b0, n, list, (T *)u,
                       (const T *)(sizeof(T) == 8 ? rhoh : rho), T(h2), colour, hom);
            ++g_launches;
            return;
        }
    }
    using S = SmCfg<D, M, T>;
    const size_t smem = S::smem();
    auto k = k_smooth<D, M, T>;
    launch_pdl(k, grid_for(k, smem, (n + S::BPC - 1) / S::BPC), smem, c.stream, A, b0, n, list, (T *)u,
               (const T *)(rhoh ? rhoh : rho), T(h2), colour, hom, rhoh ? 1 : 0);
    ++g_launches;
}

// Whole-box kernels: the cp.async-staged versions wherever a half-row holds
// a 16-byte vector (all boxes of 8^D and 16^D cells, FP64 4^D), the
// table-driven ones otherwise.
template <int D, int M, int MP, typename T>
void do_resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                       double ih2, int hom) {
    if (n <= 0) return;
    if constexpr (FpCfg<D, M, T>::ok) {
        auto go = [&](auto many) {
            constexpr bool MANY = decltype(many)::value;
            using F = FpCfg<D, M, T, rr_threads<D, M, T>(MANY)>;
            const size_t smem = F::smem();
            auto k = k_resid_restrict_p<D, M, MP, T, MANY>;
            launch_pdl(k, grid_for(k, smem, (n + F::BPC - 1) / F::BPC), smem, c.stream, A, b0, n, (T *)u, (T *)rho,
                       (T *)vold, T(ih2), hom);
        };
        if constexpr (rr_threads<D, M, T>(true) != rr_threads<D, M, T>(false)) {
            if (n > kThreads / 32 * sm_count()) go(std::true_type{});
            else go(std::false_type{});
        } else {
            go(std::false_type{});
        }
    } else {
        const size_t smem = FullCfg<D, M, T>::smem();
        auto k = k_resid_restrict<D, M, MP, T>;
        launch_pdl(k, grid_for(k, smem, work_ctas<D, M>(n)), smem, c.stream, A, b0, n, (T *)u, (T *)rho,
                   (T *)vold, T(ih2), hom);
    }
    ++g_launches;
}

template <int D, int M, typename T>
void do_fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold, double ih2,
            int hom, void *rhoh) {
    if (n <= 0) return;
    const T chat = T(-1.0 / (ih2 * 2 * D));  // -h^2 / (2D)
    if constexpr (FpCfg<D, M, T>::ok) {
        using F = FpCfg<D, M, T, fas_threads<D, M, T>()>;
        const size_t smem = F::smem();
        auto k = k_fas_p<D, M, T>;
        launch_pdl(k, grid_for(k, smem, (n + F::BPC - 1) / F::BPC), smem, c.stream, A, b0, n, (const T *)u,
                   (T *)rho, (T *)vold, T(ih2), hom, (T *)rhoh, chat);
    } else {
        const size_t smem = FullCfg<D, M, T>::smem();
        auto k = k_fas<D, M, T>;
        launch_pdl(k, grid_for(k, smem, work_ctas<D, M>(n)), smem, c.stream, A, b0, n, (const T *)u, (T *)rho,
                   (T *)vold, T(ih2), hom, (T *)rhoh, chat);
    }
    ++g_launches;
}

template <int D, int M, int MP, typename T>
void do_correct(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold) {
    if (n <= 0) return;
    // one CTA per parent: the parent staged once for its 2^D children
    if constexpr (PpCfg<D, M, T>::ok && MP == M) {
        if (c.sibs) {
            using S = PpCfg<D, M, T>;
            const size_t smem = S::smem();
            auto k = k_correct_pp<D, M, T>;
            launch_pdl(k, grid_for(k, smem, (n / S::NC + S::BPC - 1) / S::BPC), smem, c.stream, A, b0, n, (T *)u,
                       (const T *)vold);
            ++g_launches;
            return;
        }
    }
    // staged copies; in 3D the pair sums of a coarse cell are shared by its children
    if constexpr (CpCfg<D, M, T>::ok && MP == M) {
        using S = CpCfg<D, M, T>;
        const size_t smem = S::smem();
        auto k = k_correct_p<D, M, MP, T>;
        launch_pdl(k, grid_for(k, smem, (n + S::BPC - 1) / S::BPC), smem, c.stream, A, b0, n, (T *)u,
                   (const T *)vold);
        ++g_launches;
        return;
    }
    const size_t smem = CorrCfg<D, M>::template smem<T>();
    auto k = k_correct<D, M, MP, T>;
    launch_pdl(k, grid_for(k, smem, work_ctas<D, M>(n)), smem, c.stream, A, b0, n, (T *)u, (const T *)vold);
    ++g_launches;
}

template <int D, int M, int MP, typename T>
void do_restrict_u(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u) {
    if (n <= 0) return;
    auto k = k_restrict_u<D, M, MP, T>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, b0, n, list, (T *)u);
    ++g_launches;
}

template <int D, int M, typename T>
void do_leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u, const void *rho,
                      int hom, unsigned long long *rmax, unsigned long long *pmax, void *rout,
                      bool rout_f32) {
    if (n <= 0) return;
    auto go = [&](auto k, size_t smem, int wc, auto *out) {
        launch_pdl(k, grid_for(k, smem, wc), smem, c.stream, A, list, n, (const T *)u, (const T *)rho, hom, rmax,
                   pmax, out);
    };
    if constexpr (FpCfg<D, M, T>::ok) {
        using F32 = FpCfg<D, M, T, leaf_threads<D, M, T, float>()>;
        using F64 = FpCfg<D, M, T, leaf_threads<D, M, T, double>()>;
        auto k32 = c.one_tree ? k_leaf_residual_p<D, M, T, float, true> : k_leaf_residual_p<D, M, T, float, false>;
        auto k64 = c.one_tree ? k_leaf_residual_p<D, M, T, double, true> : k_leaf_residual_p<D, M, T, double, false>;
        if (rout_f32) go(k32, F32::smem(), (n + F32::BPC - 1) / F32::BPC, (float *)rout);
        else go(k64, F64::smem(), (n + F64::BPC - 1) / F64::BPC, (double *)rout);
    } else {
        const size_t smem = FullCfg<D, M, T>::smem();
        if (rout_f32) go(k_leaf_residual<D, M, T, float>, smem, work_ctas<D, M>(n), (float *)rout);
        else go(k_leaf_residual<D, M, T, double>, smem, work_ctas<D, M>(n), (double *)rout);
    }
    ++g_launches;
}

template <int D, int M, typename T>
void do_leaf_set(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *src, void *dst) {
    if (n <= 0) return;
    auto k = k_leaf_set<D, M, T>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, src, (T *)dst);
    ++g_launches;
}

template <int D, int M, typename T>
void do_leaf_get(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *src, double *dst) {
    if (n <= 0) return;
    auto k = k_leaf_get<D, M, T>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, (const T *)src, dst);
    ++g_launches;
}

template <int D, int M, int MP>
void do_bc_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, double *bc) {
    if (n <= 0) return;
    auto k = k_bc_restrict<D, M, MP>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, b0, n, bc);
    ++g_launches;
}

template <int D, int M>
void do_mixed_update(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *x, const float *e) {
    if (n <= 0) return;
    auto k = k_mixed_update<D, M>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, x, e);
    ++g_launches;
}

template <int D, int M>
void do_adjoint_apply(const LaunchCfg &c, const BoxMeta &A, const int *child, const double *hb, const int *list,
                      int n, const double *lam, double *out) {
    if (n <= 0) return;
    const size_t smem = sizeof(double) * Geo<D, M>::PC * Geo<D, M>::BPC;
    auto k = k_adjoint_apply<D, M>;
    launch_pdl(k, grid_for(k, smem, work_ctas<D, M>(n)), smem, c.stream, A, child, hb, list, n, lam, out);
    ++g_launches;
}

template <int D, int M>
void do_adjoint_db(const LaunchCfg &c, const BoxMeta &A, const double *hb, const int *list, int n, const double *lam,
                   double *db) {
    if (n <= 0) return;
    auto k = k_adjoint_db<D, M>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, hb, list, n, lam, db);
    ++g_launches;
}

template <int D, int M>
void do_axpbypcz(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *out, double a,
                 const double *x, double b, const double *y, double cc, const double *z) {
    if (n <= 0) return;
    auto k = k_leaf_axpbypcz<D, M>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, out, a, x, b, y, cc, z);
    ++g_launches;
}

template <int D, int M, typename T>
void do_precond_in(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *x, void *rho,
                   void *rhoh) {
    if (n <= 0) return;
    auto k = k_precond_in<D, M, T>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, x, (T *)rho, (T *)rhoh);
    ++g_launches;
}

template <int D, int M, typename T>
void do_precond_out(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u, double *out) {
    if (n <= 0) return;
    auto k = k_precond_out<D, M, T>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, (const T *)u, out);
    ++g_launches;
}

template <int D, int M>
void do_reduce2(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *out, double a, const double *x,
                double b, const double *y, const double *w, double *partials, double *result) {
    auto k = k_leaf_reduce2<D, M>;
    const int grid = std::min(kPartials / 2, grid_for(k, 0, std::max(1, work_ctas<D, M>(n))));
    launch_pdl(k, grid, 0, c.stream, A, list, n, out, a, x, b, y, w, partials);
    k_reduce2_final<<<1, kThreads, 0, c.stream>>>(partials, grid, out != nullptr, result);
    g_launches += 2;
}

template <int D, int M>
void do_adjoint_plain(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *lam, double *out) {
    if (n <= 0) return;
    static_assert(FpCfg<D, M, double>::ok, "leaf boxes have 4 cells per side or more");
    using F = FpCfg<D, M, double, leaf_threads<D, M, double, float>()>;
    auto k = k_adjoint_plain_p<D, M>;
    launch_pdl(k, grid_for(k, F::smem(), (n + F::BPC - 1) / F::BPC), F::smem(), c.stream, A, list, n, lam, out);
    ++g_launches;
}

template <int D, int M>
void do_reduce(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *x, const double *y,
               int mode, double *partials, double *result) {
    auto k = k_leaf_reduce<D, M>;
    const int grid = std::min(kPartials, grid_for(k, 0, std::max(1, work_ctas<D, M>(n))));
    launch_pdl(k, grid, 0, c.stream, A, list, n, x, y, mode, partials);
    k_reduce_final<<<1, kThreads, 0, c.stream>>>(partials, grid, mode, result);
    g_launches += 2;
}

template <int D, int M>
void do_rho_hat(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *rho, double *rhoh) {
    if (n <= 0) return;
    auto k = k_rho_hat<D, M>;
    launch_pdl(k, grid_for(k, 0, work_ctas<D, M>(n)), 0, c.stream, A, list, n, rho, rhoh);
    ++g_launches;
}

template <int D, typename T, bool VAR>
void do_coarse(const LaunchCfg &c, const BoxMeta &A, const CoarseArgs &G, size_t smem, int ntrees, void *u,
               const void *rho, void *vold) {
    auto k = k_coarse<D, T, VAR>;
    occupancy(reinterpret_cast<const void *>(k), smem);  // sets the shared-memory limit
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ntrees * G.R);
    cfg.blockDim = dim3(kCoarseThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = G.R;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = G.R > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, k, A, G, (T *)u, (const T *)rho, (T *)vold);
    ++g_launches;
}

// ---- dispatch over the box size --------------------------------------------
[[noreturn]] inline void bad_size(int M, int MP) {
    throw std::runtime_error("unsupported box size " + std::to_string(M) + "/" + std::to_string(MP));
}

#define AFG_SWITCH_M(M, BODY)                       \
    switch (M) {                                    \
        case 2: { constexpr int MM = 2; BODY; break; }   \
        case 4: { constexpr int MM = 4; BODY; break; }   \
        case 8: { constexpr int MM = 8; BODY; break; }   \
        case 16: { constexpr int MM = 16; BODY; break; } \
        default: bad_size(M, 0);                    \
    }

// (M, MP) pairs: same size (tree levels >= 2) or half size (root and below)
#define AFG_SWITCH_MMP(M, MP, BODY)                                                   \
    if ((M) == (MP)) {                                                                \
        switch (M) {                                                                  \
            case 4: { constexpr int MM = 4, PP = 4; BODY; break; }                    \
            case 8: { constexpr int MM = 8, PP = 8; BODY; break; }                    \
            case 16: { constexpr int MM = 16, PP = 16; BODY; break; }                 \
            default: bad_size(M, MP);                                                 \
        }                                                                             \
    } else if (2 * (MP) == (M)) {                                                     \
        switch (M) {                                                                  \
            case 4: { constexpr int MM = 4, PP = 2; BODY; break; }                    \
            case 8: { constexpr int MM = 8, PP = 4; BODY; break; }                    \
            case 16: { constexpr int MM = 16, PP = 8; BODY; break; }                  \
            default: bad_size(M, MP);                                                 \
        }                                                                             \
    } else bad_size(M, MP);

// The precision-specific launches, instantiated per (dimension, precision) in
// launch_d<D>_f64.cu / launch_d<D>_f32.cu so those compile in parallel.
template <int D, typename T>
struct PrecOps {
    static void coarse(const LaunchCfg &c, const BoxMeta &A, const CoarseArgs &G, size_t smem, int ntrees, void *u,
                       const void *rho, void *vold);
    static void smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u,
                       const void *rho, const void *rhoh, double h2, int colour, int hom);
    static void resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                               double ih2, int hom);
    static void fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold,
                    double ih2, int hom, void *rhoh);
    static void correct(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold);
    static void restrict_u(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u);
    static void leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,
                              const void *rho, int hom, unsigned long long *rmax,
                              unsigned long long *pmax, void *rout, bool rout_f32);
    static void leaf_set(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *src, void *dst);
    static void leaf_get(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *src, double *dst);
};

template <int D, typename T>
void PrecOps<D, T>::coarse(const LaunchCfg &c, const BoxMeta &A, const CoarseArgs &G, size_t smem, int ntrees, void *u,
                           const void *rho, void *vold) {
    if (G.op) do_coarse<D, T, true>(c, A, G, smem, ntrees, u, rho, vold);
    else do_coarse<D, T, false>(c, A, G, smem, ntrees, u, rho, vold);
}

template <int D, typename T>
void PrecOps<D, T>::smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u,
                           const void *rho, const void *rhoh, double h2, int colour, int hom) {
    AFG_SWITCH_M(c.M, (do_smooth<D, MM, T>(c, A, b0, n, list, u, rho, rhoh, h2, colour, hom)));
}

template <int D, typename T>
void PrecOps<D, T>::resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                                   double ih2, int hom) {
    AFG_SWITCH_MMP(c.M, c.MP, (do_resid_restrict<D, MM, PP, T>(c, A, b0, n, u, rho, vold, ih2, hom)));
}

template <int D, typename T>
void PrecOps<D, T>::fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold,
                        double ih2, int hom, void *rhoh) {
    AFG_SWITCH_M(c.M, (do_fas<D, MM, T>(c, A, b0, n, u, rho, vold, ih2, hom, rhoh)));
}

template <int D, typename T>
void PrecOps<D, T>::correct(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold) {
    AFG_SWITCH_MMP(c.M, c.MP, (do_correct<D, MM, PP, T>(c, A, b0, n, u, vold)));
}

template <int D, typename T>
void PrecOps<D, T>::restrict_u(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u) {
    AFG_SWITCH_MMP(c.M, c.MP, (do_restrict_u<D, MM, PP, T>(c, A, b0, n, list, u)));
}

template <int D, typename T>
void PrecOps<D, T>::leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,
                                  const void *rho, int hom, unsigned long long *rmax,
                                  unsigned long long *pmax, void *rout, bool rout_f32) {
    AFG_SWITCH_M(c.M, (do_leaf_residual<D, MM, T>(c, A, list, n, u, rho, hom, rmax, pmax, rout, rout_f32)));
}

template <int D, typename T>
void PrecOps<D, T>::leaf_set(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *src, void *dst) {
    AFG_SWITCH_M(c.M, (do_leaf_set<D, MM, T>(c, A, list, n, src, dst)));
}

template <int D, typename T>
void PrecOps<D, T>::leaf_get(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *src, double *dst) {
    AFG_SWITCH_M(c.M, (do_leaf_get<D, MM, T>(c, A, list, n, src, dst)));
}

template <int D>
struct DimOps {
    static void rho_hat(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *rho,
                        double *rhoh);
    static void coarse(const LaunchCfg &c, const BoxMeta &A, const CoarseArgs &G, size_t smem, int ntrees, void *u,
                       const void *rho, void *vold);
    static void smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u,
                       const void *rho, const void *rhoh, double h2, int colour, int hom);
    static void resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                               double ih2, int hom);
    static void fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold,
                    double ih2, int hom, void *rhoh);
    static void correct(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold);
    static void restrict_u(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u);
    static void leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,
                              const void *rho, int hom, unsigned long long *rmax,
                              unsigned long long *pmax, void *rout, bool rout_f32);
    static void leaf_set(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *src, void *dst);
    static void leaf_get(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *src, double *dst);
    static void bc_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, double *bc);
    static void mixed_update(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *x, const float *e);
    static void adjoint_apply(const LaunchCfg &c, const BoxMeta &A, const int *child, const double *hb,
                              const int *list, int n, const double *lam, double *out);
    static void adjoint_db(const LaunchCfg &c, const BoxMeta &A, const double *hb, const int *list, int n,
                           const double *lam, double *db);
    static void axpbypcz(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *out, double a,
                         const double *x, double b, const double *y, double cc, const double *z);
    static void precond_in(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *x, void *rho,
                           void *rhoh);
    static void precond_out(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u, double *out);
    static void reduce2(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *out, double a,
                        const double *x, double b, const double *y, const double *w, double *partials,
                        double *result);
    static void adjoint_plain(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *lam,
                              double *out);
    static void reduce(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *x,
                       const double *y, int mode, double *partials, double *result);
};

template <int D>
void DimOps<D>::coarse(const LaunchCfg &c, const BoxMeta &A, const CoarseArgs &G, size_t smem, int ntrees, void *u,
                       const void *rho, void *vold) {
    if (c.fp64) PrecOps<D, double>::coarse(c, A, G, smem, ntrees, u, rho, vold);
    else PrecOps<D, float>::coarse(c, A, G, smem, ntrees, u, rho, vold);
}

template <int D>
void DimOps<D>::smooth(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u,
                       const void *rho, const void *rhoh, double h2, int colour, int hom) {
    if (c.fp64) PrecOps<D, double>::smooth(c, A, b0, n, list, u, rho, rhoh, h2, colour, hom);
    else PrecOps<D, float>::smooth(c, A, b0, n, list, u, rho, rhoh, h2, colour, hom);
}

template <int D>
void DimOps<D>::resid_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, void *rho, void *vold,
                               double ih2, int hom) {
    if (c.fp64) PrecOps<D, double>::resid_restrict(c, A, b0, n, u, rho, vold, ih2, hom);
    else PrecOps<D, float>::resid_restrict(c, A, b0, n, u, rho, vold, ih2, hom);
}

template <int D>
void DimOps<D>::fas(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const void *u, void *rho, void *vold,
                    double ih2, int hom, void *rhoh) {
    if (c.fp64) PrecOps<D, double>::fas(c, A, b0, n, u, rho, vold, ih2, hom, rhoh);
    else PrecOps<D, float>::fas(c, A, b0, n, u, rho, vold, ih2, hom, rhoh);
}

template <int D>
void DimOps<D>::correct(const LaunchCfg &c, const BoxMeta &A, int b0, int n, void *u, const void *vold) {
    if (c.fp64) PrecOps<D, double>::correct(c, A, b0, n, u, vold);
    else PrecOps<D, float>::correct(c, A, b0, n, u, vold);
}

template <int D>
void DimOps<D>::restrict_u(const LaunchCfg &c, const BoxMeta &A, int b0, int n, const int *list, void *u) {
    if (c.fp64) PrecOps<D, double>::restrict_u(c, A, b0, n, list, u);
    else PrecOps<D, float>::restrict_u(c, A, b0, n, list, u);
}

template <int D>
void DimOps<D>::leaf_residual(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u,
                              const void *rho, int hom, unsigned long long *rmax,
                              unsigned long long *pmax, void *rout, bool rout_f32) {
    if (c.fp64) PrecOps<D, double>::leaf_residual(c, A, list, n, u, rho, hom, rmax, pmax, rout, rout_f32);
    else PrecOps<D, float>::leaf_residual(c, A, list, n, u, rho, hom, rmax, pmax, rout, rout_f32);
}

template <int D>
void DimOps<D>::leaf_set(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *src, void *dst) {
    if (c.fp64) PrecOps<D, double>::leaf_set(c, A, list, n, src, dst);
    else PrecOps<D, float>::leaf_set(c, A, list, n, src, dst);
}

template <int D>
void DimOps<D>::leaf_get(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *src, double *dst) {
    if (c.fp64) PrecOps<D, double>::leaf_get(c, A, list, n, src, dst);
    else PrecOps<D, float>::leaf_get(c, A, list, n, src, dst);
}

template <int D>
void DimOps<D>::bc_restrict(const LaunchCfg &c, const BoxMeta &A, int b0, int n, double *bc) {
    AFG_SWITCH_MMP(c.M, c.MP, (do_bc_restrict<D, MM, PP>(c, A, b0, n, bc)));
}

template <int D>
void DimOps<D>::mixed_update(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *x, const float *e) {
    AFG_SWITCH_M(c.M, (do_mixed_update<D, MM>(c, A, list, n, x, e)));
}

template <int D>
void DimOps<D>::adjoint_apply(const LaunchCfg &c, const BoxMeta &A, const int *child, const double *hb,
                              const int *list, int n, const double *lam, double *out) {
    AFG_SWITCH_M(c.M, (do_adjoint_apply<D, MM>(c, A, child, hb, list, n, lam, out)));
}

template <int D>
void DimOps<D>::adjoint_db(const LaunchCfg &c, const BoxMeta &A, const double *hb, const int *list, int n,
                           const double *lam, double *db) {
    AFG_SWITCH_M(c.M, (do_adjoint_db<D, MM>(c, A, hb, list, n, lam, db)));
}

template <int D>
void DimOps<D>::axpbypcz(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *out, double a,
                         const double *x, double b, const double *y, double cc, const double *z) {
    AFG_SWITCH_M(c.M, (do_axpbypcz<D, MM>(c, A, list, n, out, a, x, b, y, cc, z)));
}

// leaf boxes: 4, 8 or 16 cells per side
#define AFG_SWITCH_LEAF(M, BODY)                         \
    switch (M) {                                         \
        case 4: { constexpr int MM = 4; BODY; break; }   \
        case 8: { constexpr int MM = 8; BODY; break; }   \
        case 16: { constexpr int MM = 16; BODY; break; } \
        default: bad_size(M, 0);                         \
    }

template <int D>
void DimOps<D>::rho_hat(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *rho,
                        double *rhoh) {
    AFG_SWITCH_LEAF(c.M, (do_rho_hat<D, MM>(c, A, list, n, rho, rhoh)));
}

template <int D>
void DimOps<D>::precond_in(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *x, void *rho,
                           void *rhoh) {
    if (c.fp64) { AFG_SWITCH_LEAF(c.M, (do_precond_in<D, MM, double>(c, A, list, n, x, rho, rhoh))); }
    else { AFG_SWITCH_LEAF(c.M, (do_precond_in<D, MM, float>(c, A, list, n, x, rho, rhoh))); }
}

template <int D>
void DimOps<D>::precond_out(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const void *u, double *out) {
    if (c.fp64) { AFG_SWITCH_LEAF(c.M, (do_precond_out<D, MM, double>(c, A, list, n, u, out))); }
    else { AFG_SWITCH_LEAF(c.M, (do_precond_out<D, MM, float>(c, A, list, n, u, out))); }
}

template <int D>
void DimOps<D>::reduce2(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, double *out, double a,
                        const double *x, double b, const double *y, const double *w, double *partials,
                        double *result) {
    AFG_SWITCH_LEAF(c.M, (do_reduce2<D, MM>(c, A, list, n, out, a, x, b, y, w, partials, result)));
}

template <int D>
void DimOps<D>::adjoint_plain(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *lam,
                              double *out) {
    AFG_SWITCH_LEAF(c.M, (do_adjoint_plain<D, MM>(c, A, list, n, lam, out)));
}

template <int D>
void DimOps<D>::reduce(const LaunchCfg &c, const BoxMeta &A, const int *list, int n, const double *x,
                       const double *y, int mode, double *partials, double *result) {
    AFG_SWITCH_M(c.M, (do_reduce<D, MM>(c, A, list, n, x, y, mode, partials, result)));
}


}  // namespace afg
