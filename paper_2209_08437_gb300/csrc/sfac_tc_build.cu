// sfac_tc_build.cu - the dense operator of one axis and its digit image.
//
// With E_C = I + G and E_S = I + H (G circulant, H skew-circulant, both
// symmetric Toeplitz with first columns g, h) the linear factor of an axis is
//   P = (I + G)(I + H)(I + G) = I + D,  D = G + W + G W,  W = H + G + H G.
// D is formed in FP64 from the increments, so its rounding is relative to D
// itself. It runs once per plan (n = 256: 17 M multiply-adds an axis; plan creation for
// 3D 256^3 0.7 -> 1.3 ms, for 2D 1024^2 4.6 -> 9.0 ms).
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "sfac_tc.h"

namespace sfac {
namespace {

int parts_of(int n) { return n <= 128 ? 1 : 2; }
int rows_of(int n) { return n <= 128 ? n : (n + 1) / 2; }
int kp_of(int n) { return (rows_of(n) + 31) / 32 * 32; }

// First columns g, h from the expm1 values xc, xs of the spectra and cs[m] =
// cos(pi m / n):  g_d = (1/n) sum_j xc_j cos(2 pi j d / n),
// h_d = (1/n) sum_j xs_j cos(pi d (2j - 1) / n). One CTA per d; each thread sums
// with compensation (Neumaier), the partial sums are added in a fixed order.
__global__ void __launch_bounds__(128) tc_columns(int n, const double* __restrict__ spectra, double* __restrict__ g,
                                                  double* __restrict__ h) {
    const int d = blockIdx.x, skew = blockIdx.y, two_n = 2 * n;
    const double* x = spectra + skew * n;
    const double* cs = spectra + two_n;
    __shared__ double part[2][128];
    double s = 0.0, c = 0.0;
    auto add = [&](double v) {
        const double t = __dadd_rn(s, v);
        c += fabs(s) >= fabs(v) ? __dadd_rn(__dadd_rn(s, -t), v) : __dadd_rn(__dadd_rn(v, -t), s);
        s = t;
    };
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int m = (int)((skew ? (long long)d * (2 * j - 1) + two_n * (long long)n : 2LL * d * j) % two_n);
        add(__dmul_rn(x[j], cs[m]));
    }
    part[0][threadIdx.x] = s;
    part[1][threadIdx.x] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int t = 1; t < blockDim.x; ++t) {
            add(part[0][t]);
            c += part[1][t];
        }
        (skew ? h : g)[d] = (s + c) / n;
    }
}

// out = X + Y + X Y with X[i][p] = x[|i - p|]; Y = y[|p - j|] (first product) or
// the stored matrix Ym. All of them are centrosymmetric (M[i][j] =
// M[n-1-i][n-1-j]): only the first ceil(n/2) rows are formed and stored.
__global__ void __launch_bounds__(256) tc_product(int n, const double* __restrict__ x, const double* __restrict__ y,
                                                  const double* __restrict__ Ym, double* __restrict__ out) {
    const int j = blockIdx.x * 32 + threadIdx.x, i = blockIdx.y * 8 + threadIdx.y;
    const int half = (n + 1) / 2;
    if (i >= half || j >= n) return;
    double s[4] = {0, 0, 0, 0};
    for (int p0 = 0; p0 < n; p0 += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int p = p0 + q;
            if (p < n)
                s[q] = fma(x[abs(i - p)],
                           !Ym        ? y[abs(p - j)]
                           : p < half ? Ym[(size_t)p * n + j]
                                      : Ym[(size_t)(n - 1 - p) * n + (n - 1 - j)],
                           s[q]);
        }
    }
    const double yij = Ym ? Ym[(size_t)i * n + j] : y[abs(i - j)];
    out[(size_t)i * n + j] = ((s[0] + s[1]) + (s[2] + s[3])) + (x[abs(i - j)] + yij);
}

// Entry (k, j) of part p of the operator: D itself, or its action on the sums
// (p = 0) and differences (p = 1) of a line's mirrored values:
//   D x |_k = (1/2) sum_j [ E_kj (x_j + x_{n-1-j}) + O_kj (x_j - x_{n-1-j}) ].
__device__ double tc_entry(const double* D, int n, int parts, int rows, int p, int k, int j) {
    if (k >= rows || j >= rows) return 0.0;
    if (parts == 1)
        return k < (n + 1) / 2 ? D[(size_t)k * n + j] : D[(size_t)(n - 1 - k) * n + (n - 1 - j)];
    const double a = D[(size_t)k * n + j];
    const double b = D[(size_t)k * n + (n - 1 - j)];
    const bool mid_j = j == n - 1 - j, mid_k = k == n - 1 - k;
    if (p == 0) return mid_j ? a : a + b;
    return (mid_j || mid_k) ? 0.0 : a - b;
}

__global__ void __launch_bounds__(256) tc_max(int n, int parts, int rows, const double* __restrict__ D,
                                              unsigned long long* out) {
    double m = 0.0;
    const int total = parts * rows * rows;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int p = t / (rows * rows), r = t % (rows * rows);
        m = fmax(m, fabs(tc_entry(D, n, parts, rows, p, r / rows, r % rows)));
    }
    atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// Digits of every entry (NS places of B bits), written as 8 KB blocks of 128 rows x
// 32 columns: core matrices of 8 rows x 8 columns, rows first. Order of the
// blocks, the order in which a CTA streams them: (part, 32 columns, place) up to
// 256 points, (128 rows, 32 columns, part, place) above. One CTA per (row,
// part); report as in tc_build.
__global__ void __launch_bounds__(128) tc_digits(int n, int parts, int rows, int kp, const double* __restrict__ D,
                                                 const unsigned long long* __restrict__ maxbits, int NS, int B,
                                                 __half* __restrict__ img, int* report) {
    const int row = blockIdx.x, p = blockIdx.y, nkc = kp / 32;
    const double m = __longlong_as_double((long long)*maxbits);
    int f = 0;
    if (m > 0.0) {
        f = ilogb(m) + 1;  // m < 2^f: the top digit has one bit more
        f = f < -200 ? -200 : f;
    }
    if (row == 0 && p == 0 && threadIdx.x == 0) report[0] = f;
    __shared__ int sum[kTcSlices];
    __shared__ unsigned long long total;
    if (threadIdx.x == 0) total = 0;
    for (int g0 = 0; g0 < kp; g0 += 128) {
        __syncthreads();
        if (threadIdx.x < kTcSlices) sum[threadIdx.x] = 0;
        __syncthreads();
        const int j = g0 + threadIdx.x;
        if (j < kp) {
            const double v = tc_entry(D, n, parts, rows, p, row, j);
            atomicAdd(&total, (unsigned long long)(fabs(scalbn(v, 20 - f))));
            long long F = __double2ll_rn(scalbn(v, B * NS - f));
            for (int i = 0; i < NS; ++i) F += 1LL << (B * i + B - 1);
            for (int q = 0; q < NS; ++q) {  // q = 0: most significant
                const int sh = B * (NS - 1 - q);
                int d = (int)(F >> sh);
                if (q > 0) d &= (1 << B) - 1;
                d -= 1 << (B - 1);
                const size_t block = n <= kTcMaxN ? ((size_t)p * nkc + j / 32) * NS + q
                                                  : (((size_t)(row / 128) * nkc + j / 32) * 2 + p) * NS + q;
                img[block * (128 * 32) + (size_t)((j % 32) / 8) * (128 * 8) + (row % 128 / 8) * 64 + (row % 8) * 8 +
                    j % 8] = __int2half_rn(d);
                if (d) atomicAdd(&sum[q], abs(d));
            }
        }
        __syncthreads();
        if (threadIdx.x < kTcSlices) atomicMax(&report[1 + threadIdx.x], sum[threadIdx.x]);
    }
    if (threadIdx.x == 0) atomicMax(&report[1 + kTcSlices], (int)(total >> 10));
}

}  // namespace

size_t tc_image_bytes(int n, int slices) { return (size_t)parts_of(n) * ((rows_of(n) + 127) / 128) * (kp_of(n) / 32) * slices * 8192; }
size_t tc_scratch_bytes(int n) { return 2 * sizeof(double) * ((size_t)((n + 1) / 2) * n + n) + 64; }

cudaError_t tc_build(int n, int slices, int bits, const double* spectra, void* img, void* scratch, int* report_host,
                     cudaStream_t s) {
    const int parts = parts_of(n), rows = rows_of(n), kp = kp_of(n);
    double* W = static_cast<double*>(scratch);
    double* D = W + (size_t)((n + 1) / 2) * n;
    double* g = D + (size_t)((n + 1) / 2) * n;
    double* h = g + n;
    unsigned long long* mx = reinterpret_cast<unsigned long long*>(h + n);
    int* report = reinterpret_cast<int*>(mx + 1);
    cudaError_t err = cudaMemsetAsync(mx, 0, 64, s);
    if (err != cudaSuccess) return err;
    const dim3 grid((n + 31) / 32, ((n + 1) / 2 + 7) / 8), block(32, 8);
    tc_columns<<<dim3(n, 2), 128, 0, s>>>(n, spectra, g, h);
    tc_product<<<grid, block, 0, s>>>(n, h, g, nullptr, W);
    tc_product<<<grid, block, 0, s>>>(n, g, nullptr, W, D);
    tc_max<<<std::max(1, std::min(64, n / 4)), 256, 0, s>>>(n, parts, rows, D, mx);
    tc_digits<<<dim3((rows + 127) / 128 * 128, parts), 128, 0, s>>>(n, parts, rows, kp, D, mx, slices, bits, static_cast<__half*>(img),
                                             report);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    return cudaMemcpyAsync(report_host, report, (2 + kTcSlices) * sizeof(int), cudaMemcpyDeviceToHost, s);
}

bool tc_accept(int n, int slices, const void* img, const int* report, TcAxis* ax) {
    constexpr int NS = kTcSlices, B = kTcBits;
    ax->n = n;
    ax->parts = parts_of(n);
    ax->rows = rows_of(n);
    ax->kp = kp_of(n);
    ax->scale = report[0];
    ax->headroom = 0;
    if (slices != kTcSlices) {
        // FP32: the sums are rounded to 24 bits like any FP32 sum. With entries of 1/2
        // and more (long steps: D cancels most of x) the FFT passes are the more
        // accurate ones; a tiny f would leave the exponent range of the closing products.
        if (report[0] > -1 || report[0] < -60) return false;
        ax->img = img;
        return true;
    }
    // Largest sum the accumulator of order s = i + j can reach: digits of x are at
    // most 2^(B-1) in size, the top one 2^B (over 128 columns), or 2^(B-1) too if lines are scaled by
    // one more bit. Orders up to 5 must stay within 2^24 (FP32 holds every integer
    // of that size), order 6 within 2^25 and order 7 anywhere: a unit lost there is
    // below 2^-56 of the line's largest value.
    int headroom = -1;
    for (int h = 0; h < 2 && headroom < 0; ++h) {
        bool ok = true;
        for (int s = 2; s <= 6; ++s) {
            double bound = std::ldexp((double)report[s - 1], B - h);
            for (int j = 1; j < s - 1; ++j) bound += std::ldexp((double)report[j], B - 1);
            ok = ok && bound <= std::ldexp(1.0, s <= 5 ? 24 : 25);
        }
        if (ok) headroom = h;
    }
    if (headroom < 0) return false;
    // a row's sum of |entries| / 2^f, so that the 64-bit sums of the pass cannot overflow
    if (report[1 + NS] > 4 << 10 || report[0] > 2) return false;
    ax->headroom = headroom;
    ax->img = img;
    return true;
}

}  // namespace sfac
