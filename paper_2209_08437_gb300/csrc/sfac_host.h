// sfac_host.h - host-side FP64 precompute shared by plans and batches.
#pragma once

#include <vector>

namespace sfac {

// The FP64 tables of one axis (Sec. 2.1, Sec. 2.2, Remark 1).
struct AxisHost {
    int n = 0;
    std::vector<double> bcol, cfirst, sfirst, lambda, mu;
    std::vector<double> eC, eS, twist, twid;  // twist, twid: interleaved complex
    std::vector<double> incC, incS;           // e^{tau/2 lambda} - 1, e^{tau mu} - 1
    std::vector<double> dC, dS;               // the same over n, for the FP32 increment passes
};

bool is_pow2(int v);

// Smallest power of two >= 2n - 1 (at least 4).
int padded_length(int n);

// First columns of e^{tau/2 C} - I and e^{tau S} - I (both symmetric Toeplitz, n
// values each) of the axis in T.
void increment_columns(const AxisHost& T, std::vector<double>* g, std::vector<double>* h);

// The n expm1 values of each spectrum (e^{tau/2 C} - I, then e^{tau S} - I) and
// cos(pi m / n) for m = 0 .. 2n - 1, from which the columns are summed.
std::vector<double> increment_spectra(const AxisHost& T);

// Zero-padded form of one axis, for any n (needs the spectra of compute_axis in T):
// e^{t C} and e^{tau S} are symmetric Toeplitz matrices, so each is a linear
// convolution of the line with its first column; padded to a power of two L >= 2n - 1
// (padded_length) the convolution is circular and its multiplier (the DFT of the
// symmetric padded column) is real.
// mC, mS: L real multipliers incl. 1/L of e^{tau/2 C} and e^{tau S}, or (increments)
// of those less the identity.
void padded_factors(const AxisHost& T, bool increments, std::vector<double>* mC, std::vector<double>* mS);
// L real multipliers incl. 1/L of B itself (diagnostics).
void padded_operator(const AxisHost& T, std::vector<double>* mB);
// L complex e^{-2 pi i m / L}, interleaved.
std::vector<double> padded_twiddles(int n);

// Tables of one axis for Riesz order alpha, interface parameter eps, step tau,
// domain [a, b] and n interior unknowns.
void compute_axis(double alpha, double eps, double tau, double a, double b, int n, AxisHost* T);

// Ratio-twiddle records of the FP64 FFT passes of length N with E values per
// thread (E <= 16; layout in sfac_fft.cuh, FftPassRatio); empty if no pass of
// span > 1 exists.
std::vector<double> ratio_twiddles(int N, int E);

}  // namespace sfac
