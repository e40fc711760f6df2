// sfac_diag.h - launchers of the diagnostic reductions (sfac_diag.cu).
#pragma once

#include <cuda_runtime.h>

#include "sfac_internal.h"

namespace sfac {

// Number of per-CTA partials one diagnostic pass over `clines` complex lines of
// FFT length N writes.
long long diag_partials_needed(long long clines, int N);

// One diagnostic pass over the lines of `a` (field of doubles or floats,
// f64_field): accumulates into out[0] the sum of x . B x over its lines, into
// out[1] (first_axis only) the sum of (u^2 - 1)^2 and into out[2] the max of
// |u|. Tables are FP64: non-padded axes mA = lambda/N, mB = mu/N with a.twist,
// a.twid FP64; zero-padded axes mA = the real multiplier of B as a padded
// linear convolution (incl. 1/L), mB unused. `partial` holds at least
// diag_partials_needed(...) entries.
cudaError_t launch_diag_axis(bool f64_field, bool padded, int N, const PassArgs& a, const double* mA,
                             const double* mB, int first_axis, double3* partial, double* out, cudaStream_t s);

// Small grids: every line of every axis by one CTA of one launch, x . B x as the
// Toeplitz sum b_0 sum x_i^2 + 2 sum_d b_d sum_i x_i x_{i+d}, and the final sum by
// the CTA that finishes last (fixed order).
struct DiagDirect {
    const void* u;
    int dim;
    int n[3];
    long long inner[3], lines[3];
    const double* b[3];     // first column of B_axis
    double3* partial;       // one entry per line of all axes
    unsigned int* counter;  // arrivals, modulo the CTAs of a launch: 0 before and after
    double* out;            // out[0..2] as launch_diag_axis
};
// (for grids that diag_direct_pays admits: lines of at most 1024 points)
cudaError_t launch_diag_direct(bool f64_field, const DiagDirect& d, cudaStream_t s);

}  // namespace sfac
