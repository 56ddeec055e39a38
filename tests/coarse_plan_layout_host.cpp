// Host harness for the shared-memory layout of csrc/coarse_plan.h, with and
// without variable coefficients: what the coarse launch reads and writes lies in
// the block's memory, apart from everything else, aligned for its copies; prints
// the number of plans and of failed checks.
#include <algorithm>
#include <cstdio>

#include "../paper_1701_04329_gb300/csrc/coarse_plan.h"

int main() {
    using namespace afg;
    int plans = 0, bad = 0;
    auto check = [&](bool ok) { bad += !ok; };
    const int roots[][3] = {{1, 1, 1}, {3, 2, 1}, {5, 3, 1}, {1, 1, 6}, {2, 1, 3}, {1, 7, 1}};
    for (int D = 2; D <= 3; ++D)
        for (int fp64 = 0; fp64 < 2; ++fp64)
            for (int N : {4, 8, 16})
                for (int M = 2; M <= (D == 2 ? 256 : 32); M *= 2)
                    for (const auto &nr : roots)
                        for (int T : {1, 7})
                            for (int var = 0; var < 2; ++var) {
                                CoarseArgs G;
                                const size_t es = fp64 ? 8 : 4, bytes = coarse_plan(D, fp64, M, N, nr, T, G, var);
                                ++plans;
                                const size_t head = (sizeof(CoarseArgs) + 15) / 16 * 16;
                                check(bytes >= head + (size_t)G.total * es + 9u * G.slab_boxes);
                                int scratch = 0, end = 0;
                                auto padded = [&](int li) {
                                    return (G.P[li] + 2) * (G.nx[li] + 2) * (D == 3 ? G.ny[li] + 2 : 1);
                                };
                                for (int li = 0; li + 1 < G.nl; ++li) scratch = std::max(scratch, padded(li));
                                check(G.total >= G.odc + scratch);  // the correction's differences of any level below the top
                                // boxes of the top level that a block's slab touches: cell0[] and refined[] hold one entry each
                                const int lt = G.nl - 1, layer = D == 3 ? G.nbx * G.nby : G.nbx;
                                for (int r = 0; r < G.R; ++r) {
                                    const int z0 = G.nr[lt] > 1 ? r * G.P[lt] : 0;
                                    const int first = (z0 >> G.lgmb) * layer;
                                    check((((z0 + G.P[lt] - 1) >> G.lgmb) + 1) * layer - first <= G.slab_boxes);
                                }
                                if (!var) {
                                    check(G.ncoef == 0);
                                    continue;
                                }
                                // coefficients: behind the grids (cleared up to ocoef), level after level, 16-byte pieces
                                check(G.ocoef >= G.odc + scratch && G.ocoef % 4 == 0 && G.ncoef % 4 == 0);
                                check(G.ocoef * es % 16 == 0 && G.ncoef * es % 16 == 0 && head % 16 == 0);
                                end = G.ocoef;
                                for (int li = 0; li < G.nl; ++li) {
                                    check(G.oc[li] >= end && G.csz[li] >= padded(li));
                                    end = G.oc[li] + (2 * D + 2) * G.csz[li];
                                }
                                check(end <= G.ocoef + G.ncoef && G.ocoef + G.ncoef <= G.total);
                            }
    std::printf("%d %d\n", plans, bad);
    return bad != 0;
}
