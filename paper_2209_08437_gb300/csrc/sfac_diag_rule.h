// sfac_diag_rule.h - which grids take the one-launch diagnostics (host only).
#pragma once

namespace sfac {

// Whether the direct Toeplitz sums of a grid (diag_direct_kernel: one launch, a CTA
// for each line of each axis) are expected to take no longer than the FFT passes
// (a launch and a reduction an axis, which are latency bound on such grids).
// fft_len, padded: the FFT passes of the axes.
//
// Both times are estimates in microseconds of a whole call, fitted to 246 grids
// timed both ways side by side on GB300. The direct sums cost about 1/140 us a
// CTA and the FP64 work, and no less than the longest line on one SM: its
// offsets go in rounds of 128, n = 512 50 us, n = 1024 190 us, n = 2048 720 us
// (twice as much where those CTAs come last and share SMs). Under a rule that
// bounded the work alone, 2048 x 8 took 774 us instead of 148, 1024 x 32 224
// instead of 105, 3 x 114 x 256 249 instead of 108. Under this one the direct
// sums are at most 1.08 times as long as the FFT passes on those grids, and the
// FFT passes at most 1.3 times as long as the direct sums.
inline bool diag_direct_pays(int dim, const int* n, const int* fft_len, const bool* padded) {
    double points = 1.0;
    int longest = 0;
    for (int l = 0; l < dim; ++l) {
        points *= n[l];
        longest = n[l] > longest ? n[l] : longest;
    }
    if (longest > 1024) return false;
    double lines = 0.0, work = 0.0, fft = 34.0 + 1.5e-4 * points;
    for (int l = 0; l < dim; ++l) {
        const int N = fft_len[l];
        lines += points / n[l];
        work += 0.5 * points * n[l];
        fft += padded[l] ? (N <= 1024 ? 17.0 : N == 2048 ? 39.0 : 89.0)
                         : (N <= 16 ? 19.0 : N <= 32 ? 26.0 : N <= 256 ? 29.0 : N <= 1024 ? 36.0 : 82.0);
    }
    if (work > 2.4e7) return false;  // the range of the measurements
    const double line = 0.0225 * ((longest + 127) / 128) * longest;
    const double tail = dim == 3 && n[2] == longest ? 0.9 * line : 0.0;
    return 30.0 + lines / 140.0 + 1.5e-6 * work + line + tail <= fft;
}

}  // namespace sfac
