// Host harness for the exponent an image is aligned to and the sums formed on it
// (csrc/fxsum.cuh).  Per group on stdin: the operator (h half-sweep in 3D, l and m
// the operator in 3D and 2D, r the restriction in 3D) and its values as bit
// patterns; prints the exponent (-1: not aligned), the rounded sums on the aligned
// values and the sums that are formed without alignment.
#include <cinttypes>
#include <cmath>
#include <cstdio>

#include "../paper_1701_04329_gb300/csrc/fxsum.cuh"

using namespace afg;

static void put(double x) { std::printf(" %016" PRIx64, fx_bits(x)); }

// x[0]: the centre, weight -K; then K neighbours
template <int W, int K>
static void lap(const double *x, int E, bool centre) {
    int64_t S = centre ? -K * fx_align<W>(x[0], E) : 0;
    for (int i = 1; i <= K; ++i) S += fx_align<W>(x[i], E);
    put(fx_round<W>(S, E));
}

// what the kernels form where a box is not aligned: four neighbours (and the centre) exactly, then FP64 additions
template <int K, int C>
static void plain(const double *x) {
    double s;
    if (!fx_sum<4, C>(x + 1, x[0], s)) s = std::fma(-double(C), x[0], (x[1] + x[2]) + (x[3] + x[4]));
    for (int i = 5; i <= K; ++i) s += x[i];
    put(s);
}

int main() {
    char op;
    while (std::scanf(" %c", &op) == 1) {
        const int n = op == 'r' ? 32 : op == 'm' ? 5 : 7;
        double x[32];
        uint32_t mx = 0, mn = 0xffffffffu;
        for (int i = 0; i < n; ++i) {
            uint64_t b;
            if (std::scanf("%" SCNx64, &b) != 1) return 1;
            x[i] = fx_double(b);
            fx_fold(x[i], mx, mn);
        }
        const int E = op == 'h' ? fx_common_exponent<6>(mx, mn) : op == 'l' ? fx_common_exponent<12>(mx, mn)
                    : op == 'm' ? fx_common_exponent<8>(mx, mn) : fx_common_exponent<48>(mx, mn);
        std::printf("%d", E);
        const int e = E < 0 ? kFxEmin : E;
        if (op == 'h') lap<6, 6>(x, e, false), plain<6, 0>(x);
        if (op == 'l') lap<12, 6>(x, e, true), plain<6, 6>(x);
        if (op == 'm') lap<8, 4>(x, e, true), plain<4, 4>(x);
        if (op == 'r') {  // eight children, then their 24 outer neighbours: the means of u and of h^2 A u
            int64_t su = 0, so = 0;
            double pu = 0, po = 0;
            for (int i = 0; i < 8; ++i) su += fx_align<48>(x[i], e), pu += x[i];
            for (int i = 8; i < 32; ++i) so += fx_align<48>(x[i], e), po += x[i];
            put(fx_round<48>(su, e - 3)), put(fx_round<48>(so - 3 * su, e - 3));
            put(pu / 8), put(std::fma(-3.0, pu, po) / 8);
        }
        std::printf("\n");
    }
    return 0;
}
