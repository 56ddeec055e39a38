// Host harness for csrc/coarse_plan.h: for every plan of the command line's
// sweep, the division constants, the shared-memory layout and the face slots
// are checked; prints the number of plans and of failed checks.
#include <cstdio>
#include <set>

#include "../paper_1701_04329_gb300/csrc/coarse_plan.h"

static int div_by(unsigned c, unsigned magic) {
    return magic ? (int)(((unsigned long long)c * magic) >> 32) : (int)c;
}

int main() {
    using namespace afg;
    int plans = 0, bad = 0;
    const int roots[][3] = {{1, 1, 1}, {3, 2, 1}, {5, 3, 1}, {1, 1, 6}, {2, 1, 3}};
    for (int D = 2; D <= 3; ++D)
        for (int fp64 = 0; fp64 < 2; ++fp64)
            for (int N : {4, 8, 16})
                for (int M = 2; M <= (D == 2 ? 256 : 32); M *= 2)
                    for (const auto &nr : roots)
                        for (int T : {1, 7}) {
                            CoarseArgs G;
                            const size_t bytes = coarse_plan(D, fp64, M, N, nr, T, G);
                            ++plans;
                            auto check = [&](bool ok) { bad += !ok; };
                            int end = 0;
                            for (int li = 0; li < G.nl; ++li) {
                                const int ny = D == 3 ? G.ny[li] : 1, plane = G.nx[li] / 2 * ny;
                                const int size = (G.P[li] + 2) * (G.nx[li] + 2) * (D == 3 ? ny + 2 : 1);
                                check(G.P[li] * G.nr[li] == (D == 3 ? nr[2] : nr[1]) * (2 << li));
                                check(G.nr[li] == 1 || (G.nr[li] == G.R && G.P[li] % 2 == 0 && T == 1));
                                check(li == 0 || G.nr[li] >= G.nr[li - 1]);
                                check(G.ou[li] >= end && G.orh[li] >= G.ou[li] + size && G.ov[li] >= G.orh[li] + size);
                                end = G.ov[li] + (li + 1 < G.nl ? size : 0);
                                check(G.ng[li] >= 1 && (G.ng[li] == 1 || G.ng[li] * plane <= kCoarseThreads));
                                const unsigned most = (unsigned)(2 * plane * G.P[li]) + kCoarseThreads;
                                for (unsigned c = 0; c < most; c += c < 4096 ? 1 : 37) {
                                    check(div_by(c, G.mh[li]) == (int)(c / (G.nx[li] / 2)));
                                    check(div_by(c, G.mx[li]) == (int)(c / G.nx[li]));
                                    check(div_by(c, G.mp[li]) == (int)(c / plane));
                                    if (D == 3) check(div_by(c, G.my[li]) == (int)(c / ny));
                                }
                            }
                            check(G.odc >= end && G.total >= G.odc);
                            check(bytes >= sizeof(CoarseArgs) + (size_t)G.total * (fp64 ? 8 : 4) + 9u * G.slab_boxes);
                            for (int r = 0; r < G.R; ++r)
                                for (int pm : {0, 1, 2, (1 << D) - 1}) {
                                    const std::vector<int> f = coarse_faces(D, G, r, pm);
                                    std::set<int> once(f.begin(), f.end());
                                    check(once.size() == f.size());
                                    for (int q : f) check(q >= 0 && q < G.total);
                                }
                        }
    std::printf("%d %d\n", plans, bad);
    return bad != 0;
}
