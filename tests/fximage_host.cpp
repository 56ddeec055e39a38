// Host harness for the aligned images of csrc/fxsum.cuh: reads doubles (bit
// patterns) from stdin, groups of 7 (centre, then six neighbours), each with the
// exponent to align to, and prints the rounded sum of the neighbours less six
// times the centre; or, in mode "f", single doubles as floats.
#include <cinttypes>
#include <cstdio>
#include <cstring>

#include "../paper_1701_04329_gb300/csrc/fxsum.cuh"

int main(int argc, char **argv) {
    using namespace afg;
    uint64_t b[7];
    if (argc > 1 && argv[1][0] == 'f') {
        while (std::scanf("%" SCNx64, &b[0]) == 1) {
            const float f = fx_to_float(fx_double(b[0]));
            uint32_t o;
            std::memcpy(&o, &f, 4);
            std::printf("%08x\n", o);
        }
        return 0;
    }
    if (argc > 1 && argv[1][0] == 'd') {
        uint32_t f;
        while (std::scanf("%" SCNx32, &f) == 1) {
            float x;
            std::memcpy(&x, &f, 4);
            std::printf("%016" PRIx64 "\n", fx_bits(fx_to_double(x)));
        }
        return 0;
    }
    int E;
    while (std::scanf("%d", &E) == 1) {
        for (int i = 0; i < 7; ++i)
            if (std::scanf("%" SCNx64, &b[i]) != 1) return 1;
        int64_t S = -6 * fx_align<12>(fx_double(b[0]), E);
        for (int i = 1; i < 7; ++i) S += fx_align<12>(fx_double(b[i]), E);
        std::printf("%016" PRIx64 "\n", fx_bits(fx_round<12>(S, E)));
    }
    return 0;
}
