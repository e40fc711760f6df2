// Host check of the contiguous loads of the tensor-core passes (tc_load8 in
// csrc/sfac_tc_tile.cuh and sfac_tc_tile_f32.cuh): for every length with such a
// pass, few lines and every start of the field within a group of four values,
// the values that the eight-value loads read stay inside the field. Prints
// "<loads> <grouped>": how many loads there were, how many as whole groups.
#include <cstdio>

#include "sfac_tc.h"

using namespace sfac;

int main() {
    long long loads = 0, grouped = 0;
    for (int n = kTcMinN; n <= kTcMaxN; ++n)
        for (long long lines = 1; lines <= 6; ++lines)
            for (int phase = 0; phase < 4; ++phase) {
                const long long total = lines * n;
                const int parts = n <= 128 ? 1 : 2, rows = parts == 1 ? n : (n + 1) / 2;
                for (long long L = 0; L < lines; ++L)
                    for (int c = 0; 8 * c + 8 <= rows; ++c)
                        for (int mirrored = 0; mirrored < parts; ++mirrored) {
                            const long long i = L * n + (mirrored ? n - 8 - 8 * c : 8 * c);
                            const int s = (int)((phase + i) & 3);
                            long long first = i, last = i + 8;
                            ++loads;
                            if (s == 0 || tc_groups_inside(i, total)) {
                                first = i - s;
                                last = s == 0 ? i + 8 : i - s + 12;
                                ++grouped;
                            }
                            if (first < 0 || last > total) {
                                std::printf("outside: n %d lines %lld phase %d line %lld chunk %d\n", n, lines, phase, L, c);
                                return 1;
                            }
                            if (L > 0 && L + 1 < lines && first == i && last == i + 8 && s != 0) {
                                std::printf("narrow: n %d lines %lld phase %d line %lld chunk %d\n", n, lines, phase, L, c);
                                return 1;
                            }
                        }
            }
    std::printf("%lld %lld\n", loads, grouped);
    return 0;
}
