// Prints "1" or "0" for each grid read from stdin ("dim n1 .. nd", then the FFT
// length and the padded flag of each axis): whether diag_direct_pays admits it.
#include <cstdio>

#include "sfac_diag_rule.h"

int main() {
    int dim;
    while (std::scanf("%d", &dim) == 1) {
        int n[3], len[3];
        bool padded[3];
        for (int l = 0; l < dim; ++l)
            if (std::scanf("%d", &n[l]) != 1) return 1;
        for (int l = 0; l < dim; ++l) {
            int p;
            if (std::scanf("%d %d", &len[l], &p) != 2) return 1;
            padded[l] = p != 0;
        }
        std::printf("%d\n", sfac::diag_direct_pays(dim, n, len, padded) ? 1 : 0);
    }
    return 0;
}
