// sfac_tc.h - axis passes as exact digit products on the tensor cores.
#pragma once

#include <cuda_runtime.h>

#include "sfac_internal.h"
#include "sfac_steps.h"

namespace sfac {

// The linear factor of one axis as a dense operator D = P - I, cut into
// fixed-point digits (see sfac_tc_tile.cuh). `img` holds the digit blocks in the
// order the pass streams them.
struct TcAxis {
    const void* img = nullptr;  // NULL: the axis has no tensor-core pass
    int n = 0;                  // line length
    int parts = 0;              // 1: D itself; 2: its even and odd halves
    int rows = 0;               // rows (outputs) per part: n, or ceil(n/2)
    int kp = 0;                 // rows rounded up to a multiple of 32 (K of the products)
    int scale = 0;              // exponent f: the entries are below 2^f in size
    int headroom = 0;           // more bits above a line's largest value (0 or 1)
};

// Digits per operand entry, and their width in bits: FP64, FP32.
constexpr int kTcSlices = 6, kTcBits = 9;
constexpr int kTcSlices32 = 3, kTcBits32 = 10;
// Lengths with a tensor-core pass.
constexpr int kTcMinN = 17, kTcMaxN = 256;
// FP64 lines above kTcMaxN take clusters of CTAs (sfac_tc_long.cu).
constexpr int kTcLongMaxN = 1024;

// Whether the passes may load the eight values from index i of a field of `total`
// values as whole aligned groups of four (32-byte sectors of FP64, 16 bytes of
// FP32). Where the values start inside a group, three groups hold them: up to
// three values before and three after are read too, which at the field's ends
// are somebody else's memory.
__host__ __device__ constexpr bool tc_groups_inside(long long i, long long total) { return i >= 3 && i + 11 <= total; }

// Device bytes of the digit image of an axis of n points, and of the scratch
// the builder needs for it.
size_t tc_image_bytes(int n, int slices);
size_t tc_scratch_bytes(int n);

// What the builder says of an operator, in device memory that is zero before. The
// products of a row and 128 columns are summed in one accumulator per order s = i + j
// of the digit places, s = 2..6 here; sums[h][s - 2] is the largest over all rows and
// column groups of what that accumulator can reach, in units of 2^(B - 1), with the
// top digit of the lines at most 2^B (h = 0) or 2^(B - 1) (h = 1).
struct TcReport {
    unsigned long long largest;  // bits of the largest |entry|
    int scale;                   // exponent f: the entries are below 2^f
    int row_sum;                 // largest row sum of |entries| in units of 2^(f - 10)
    int sums[2][5];
};

struct TcBuildAxis {
    int n;
    const double* spectra;  // increment_spectra's 4n values (device)
    void* img;              // tc_image_bytes
    TcReport* report;
};

// Builds the images of `count` (at most 3) axes on stream s; scratch: the sum of
// their tc_scratch_bytes.
cudaError_t tc_build(int count, const TcBuildAxis* axes, int slices, int bits, void* scratch, cudaStream_t s);

// Fills *ax from the builder's report; false where the sums could leave the
// range in which the products are exact (the axis then keeps its FFT pass).
bool tc_accept(int n, int slices, const void* img, const TcReport& report, TcAxis* ax);

// One axis pass (the arguments of launch_pass_f64 / _f32) through the tensor cores.
cudaError_t launch_pass_tc_f64(const TcAxis& ax, const PassArgs& a, cudaStream_t s);
cudaError_t launch_pass_tc_f32(const TcAxis& ax, const PassArgs& a, cudaStream_t s);

// FP64 lines of 257 to 1024 points.
cudaError_t launch_pass_tc_long(const TcAxis& ax, const PassArgs& a, cudaStream_t s);
// FP64 up to 256 points with tiles of 8 lines (few lines: latency bound).
cudaError_t launch_pass_tc_small(const TcAxis& ax, const PassArgs& a, cudaStream_t s);

// A whole call on a small grid (as launch_steps) with the operators ax[0..dim-1].
cudaError_t launch_tc_steps(const TcAxis* ax, const StepsArgs& a, cudaStream_t s);

}  // namespace sfac
