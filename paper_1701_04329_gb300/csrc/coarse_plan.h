// Plan of the coarse launch (kernels_coarse.cuh): the grids of 2, 4, ..., M
// cells per root box side, how each is held by the blocks of the cluster, and
// where it lies in shared memory.  Host and device share the struct; the plan
// is made on the host once per grid and precision.
#pragma once
#include <algorithm>
#include <cstddef>
#include <vector>

namespace afg {

constexpr int kCoarseMaxLevels = 10;  // 2 .. 1024 cells per root box side
constexpr int kCoarseThreads = 512;
constexpr int kCoarseCluster = 8;     // blocks per cluster where a tree's grids are spread (the portable size)

struct CoarseArgs {
    int nl = 0, R = 1;                // levels held, blocks per tree
    int mode = 0, nd = 0, nu = 0, nb = 0, hom = 0, fas = 0;
    int mb = 0, lgmb = 0;             // cells per box side on the top level
    int nbx = 1, nby = 1, nbz = 1;    // its boxes per axis
    int nx[kCoarseMaxLevels], ny[kCoarseMaxLevels], P[kCoarseMaxLevels], nr[kCoarseMaxLevels];
    unsigned mh[kCoarseMaxLevels], mx[kCoarseMaxLevels], my[kCoarseMaxLevels];
    int ng[kCoarseMaxLevels];         // planes relaxed side by side by one block's threads
    unsigned mp[kCoarseMaxLevels];    // division by the half-cells of a plane
    int ou[kCoarseMaxLevels], ov[kCoarseMaxLevels], orh[kCoarseMaxLevels];
    int odc = 0, total = 0;           // correction scratch, elements in all
    int slab_boxes = 0;               // top-level boxes of one block's slab (at most)
    int nface = 0;                    // faces of one block's levels on the domain sides (at most)
    const int *fslot = nullptr;       // per block of a cluster: their ghost slots, -1 past the last
    double *fval = nullptr;           // per block: their boundary values
    // variable coefficients: operator, per level its arrays (csz apart), all
    // of them contiguous, 16-byte aligned; the packed image per block, and
    // where mode 3 gathers it from
    int op = 0, N = 0;
    int oc[kCoarseMaxLevels], csz[kCoarseMaxLevels];
    int ocoef = 0, ncoef = 0;
    void *cpack = nullptr;
    const void *coef = nullptr;
    long long coef_n = 0;
    const int *dtab[kCoarseMaxLevels];  // every level's boxes by position, per tree
    const int *dbox = nullptr;        // top level's boxes by position, per tree
    const int *tree_bc = nullptr;     // per tree: Neumann sides | periodic axes << 6
};

inline unsigned coarse_magic(int d) { return d == 1 ? 0u : (unsigned)((((unsigned long long)1 << 32) + d - 1) / d); }

// Grids of 2 .. M cells per root box side for a block of nroot roots; ntrees
// blocks run side by side.  Returns the shared memory of one block in bytes.
inline size_t coarse_plan(int D, bool fp64, int M, int N, const int *nroot, int ntrees, CoarseArgs &G,
                          bool var = false) {
    G = CoarseArgs();
    G.N = N;
    G.mb = std::min(M, N);
    while ((1 << G.lgmb) < G.mb) ++G.lgmb;
    const int f = M / G.mb;
    G.nbx = nroot[0] * f;
    G.nby = nroot[1] * f;
    G.nbz = D == 3 ? nroot[2] * f : 1;
    // A grid is spread over the cluster's blocks from this many cells on: below,
    // a half-sweep costs less than the cluster barrier (350-450 cycles) that
    // spreading adds.  16^3: FP64 62 us a visit on eight blocks, 130 us on one
    // (one SM's FP64 rate); FP32 solves 1-10 % faster on eight (the 3 x 2 block
    // of roots 4.4 -> 4.0 ms, 3D gradients 16.1 -> 15.8 ms).
    const long long spread = 4096;
    size_t off = 0, dc = 0;
    for (int m = 2; m <= M; m *= 2) {
        const int li = G.nl++;
        const int nx = nroot[0] * m, ny = D == 3 ? nroot[1] * m : 1, nz = (D == 3 ? nroot[2] : nroot[1]) * m;
        const long long cells = (long long)nx * ny * nz;
        // slabs of an even number of planes, so that coarse planes do not straddle blocks
        const bool split = ntrees == 1 && cells >= spread && m >= 2 * kCoarseCluster;
        G.nx[li] = nx;
        G.ny[li] = ny;
        G.nr[li] = split ? kCoarseCluster : 1;
        G.P[li] = nz / G.nr[li];
        if (split) G.R = kCoarseCluster;
        G.mh[li] = coarse_magic(nx / 2);
        G.mx[li] = coarse_magic(nx);
        G.my[li] = coarse_magic(ny);
        G.ng[li] = std::max(1, std::min(G.P[li], kCoarseThreads / (nx / 2 * ny)));
        G.mp[li] = coarse_magic(nx / 2 * ny);
        const size_t padded = (size_t)(G.P[li] + 2) * (nx + 2) * (D == 3 ? ny + 2 : 1);
        const size_t even = (padded + 1) / 2 * 2;
        G.ou[li] = (int)off;
        off += even;
        G.orh[li] = (int)off;
        off += even;
        G.ov[li] = (int)off;
        if (2 * m <= M) {  // v' of the top level stays in global memory
            off += even;
            dc = std::max(dc, even);
        }
    }
    G.odc = (int)off;
    off += dc;
    if (var) {
        off = (off + 3) / 4 * 4;
        G.ocoef = (int)off;
        for (int li = 0; li < G.nl; ++li) {
            const size_t padded = (size_t)(G.P[li] + 2) * (G.nx[li] + 2) * (D == 3 ? G.ny[li] + 2 : 1);
            G.csz[li] = (int)((padded + 1) / 2 * 2);
            G.oc[li] = (int)off;
            off += (size_t)G.csz[li] * (2 * D + 2);
        }
        off = (off + 3) / 4 * 4;
        G.ncoef = (int)off - G.ocoef;
    }
    G.total = (int)off;
    G.slab_boxes = G.nbx * G.nby * G.nbz;
    if (G.nr[G.nl - 1] > 1) {
        const int layer = D == 3 ? G.nbx * G.nby : G.nbx;
        G.slab_boxes = std::min(G.slab_boxes, layer * (G.P[G.nl - 1] / G.mb + 2));
    }
    return (sizeof(CoarseArgs) + 15) / 16 * 16 + (off * (fp64 ? 8 : 4) + 15) / 16 * 16 + (size_t)G.slab_boxes * 9 + 16;
}

// Ghost slots of the faces on the domain sides, level by level (what a block
// of the cluster keeps in the ghost slots of its sources).  pm: periodic axes.
inline std::vector<int> coarse_faces(int D, const CoarseArgs &G, int rank, int pm) {
    std::vector<int> out;
    for (int li = 0; li < G.nl; ++li) {
        const int nx = G.nx[li], ny = D == 3 ? G.ny[li] : 1, P = G.P[li], W = nx + 2, PS = D == 3 ? W * (ny + 2) : W;
        auto slot = [&](int i, int j, int k) { return G.orh[li] + (k + 1) * PS + (D == 3 ? (j + 1) * W : 0) + i + 1; };
        for (int s = 0; s < 2 * D; ++s) {
            const int a = s >> 1, up = s & 1, last = D - 1;
            if ((pm >> a) & 1) continue;
            if (a == last) {
                if (G.nr[li] > 1 && rank != (up ? G.nr[li] - 1 : 0)) continue;
                for (int j = 0; j < ny; ++j)
                    for (int i = 0; i < nx; ++i) out.push_back(slot(i, j, up ? P : -1));
            } else if (a == 0) {
                for (int k = 0; k < P; ++k)
                    for (int j = 0; j < ny; ++j) out.push_back(slot(up ? nx : -1, j, k));
            } else {
                for (int k = 0; k < P; ++k)
                    for (int i = 0; i < nx; ++i) out.push_back(slot(i, up ? ny : -1, k));
            }
        }
    }
    return out;
}

}  // namespace afg
