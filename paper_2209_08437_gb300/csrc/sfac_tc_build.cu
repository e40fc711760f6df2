// sfac_tc_build.cu - the dense operator of one axis and its digit image.
//
// With E_C = I + G and E_S = I + H (G circulant, H skew-circulant, both
// symmetric Toeplitz with first columns g, h) the linear factor of an axis is
//   P = (I + G)(I + H)(I + G) = I + D,  D = G + W + G W,  W = H + G + H G.
// D is formed in FP64 from the increments, so its rounding is relative to D
// itself. Only its first column takes matrix-vector products. With Z the cyclic
// shift, Z E_C Z^-1 = E_C, and Z E_S Z^-1 - E_S = -2 (e_0 v^T + v e_0^T) with v = h but
// v_0 = 0 (h_{n-k} = -h_k); hence along a diagonal
//   D_{i+1,j+1} = D_{ij} + 2 (g_{i+1} w_{j+1} + w_{i+1} g_{j+1}),  w = (I + G) v.
// So D takes n^2 operations, not two products of n^3 / 2 on the FP64 pipe, and against
// 80-bit arithmetic its largest error is 1.8e-18 at n = 256 (the products: 5.9e-18).
// It runs once per plan, all axes in one set of launches (n = 1024, two axes: columns
// 52 us, vectors 28, diagonals 64, largest entry 21, digits 45). Plan creation side by
// side, with the products / now / without operators (ms): 2D 64^2 0.69 / 0.56 / 0.51,
// 255^2 1.64 / 0.84 / 1.25, 1024^2 8.99 / 4.93 / 4.70, 3D 256^3 1.45 / 0.99 / 0.93.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "sfac_tc.h"

namespace sfac {
namespace {

__host__ __device__ int parts_of(int n) { return n <= 128 ? 1 : 2; }
__host__ __device__ int rows_of(int n) { return n <= 128 ? n : (n + 1) / 2; }
__host__ __device__ int kp_of(int n) { return (rows_of(n) + 31) / 32 * 32; }

// One axis at work; its arrays but the first and the last two in the scratch.
struct TcBuild {
    int n;
    const double* spectra;
    double *g, *h, *wc, *wc_low, *w, *d0, *d0_low, *D;
    void* img;
    TcReport* report;
};
// All axes of a plan: blockIdx.z of every launch.
struct TcBuilds {
    TcBuild axis[3];
    int slices, bits;
};

// Compensated sum s + c: Knuth's branch-free two-sum collects the rounding of s in c.
struct TcSum {
    double s = 0.0, c = 0.0;
    __device__ __forceinline__ void add(double v) {
        const double t = __dadd_rn(s, v), b = __dadd_rn(t, -s);
        c = __dadd_rn(c, __dadd_rn(__dadd_rn(s, -__dadd_rn(t, -b)), __dadd_rn(v, -b)));
        s = t;
    }
};

constexpr int kTcSumThreads = 128;

// The sum over the CTA's threads, in thread 0.
__device__ double tc_cta_sum(double a) {
    __shared__ double part[kTcSumThreads / 32];
    for (int w = 16; w > 0; w >>= 1) a += __shfl_xor_sync(0xffffffffu, a, w);
    if (threadIdx.x % 32 == 0) part[threadIdx.x / 32] = a;
    __syncthreads();
    return (part[0] + part[1]) + (part[2] + part[3]);
}
__device__ double tc_cta_sum(TcSum a) {
    __shared__ double part[2][kTcSumThreads];
    const int tid = threadIdx.x;
    part[0][tid] = a.s;
    part[1][tid] = a.c;
    for (int w = kTcSumThreads / 2; w > 0; w >>= 1) {
        __syncthreads();
        if (tid < w) {
            a.add(part[0][tid + w]);
            a.c += part[1][tid + w];
            part[0][tid] = a.s;
            part[1][tid] = a.c;
        }
    }
    return a.s + a.c;
}

// First columns g, h from the expm1 values xc, xs of the spectra and cs[m] =
// cos(pi m / n):  g_d = (1/n) sum_j xc_j cos(2 pi j d / n),
// h_d = (1/n) sum_j xs_j cos(pi d (2j - 1) / n); g_{n-d} = g_d, h_{n-d} = -h_d. One
// CTA per d <= n / 2 and column.
__global__ void __launch_bounds__(kTcSumThreads) tc_columns(const __grid_constant__ TcBuilds all) {
    const TcBuild& b = all.axis[blockIdx.z];
    const int n = b.n, d = blockIdx.x, skew = blockIdx.y;
    if (2 * d > n) return;
    const unsigned two_n = 2 * n;
    const double* x = b.spectra + skew * n;
    const double* cs = b.spectra + two_n;
    TcSum a;
    for (int j = threadIdx.x; j < n; j += kTcSumThreads)
        a.add(__dmul_rn(x[j], cs[(unsigned)(skew ? d * (2 * j - 1) + d * 2 * n : 2 * d * j) % two_n]));
    double v = tc_cta_sum(a) / n;
    if (threadIdx.x != 0) return;
    if (skew && 2 * d == n) v = 0.0;
    double* column = skew ? b.h : b.g;
    column[d] = v;
    if (d > 0) column[n - d] = skew ? -v : v;
}

// a + (b + c), with the rounding of the two additions in *low.
__device__ double tc_add3(double a, double b, double c, double* low) {
    TcSum s;
    s.s = b;
    s.add(c);
    s.add(a);
    const double hi = s.s + s.c;
    *low = s.c - (hi - s.s);
    return hi;
}

// One CTA per entry i: wc = (H + G + H G) e_0 = h + g + H g and w = v + G v (see above).
// The rounding of wc, and below of D's first column, is kept: it would go into every
// entry of a diagonal alike, and from there into every step of a call.
__global__ void __launch_bounds__(kTcSumThreads) tc_vectors(const __grid_constant__ TcBuilds all) {
    const TcBuild& b = all.axis[blockIdx.z];
    const int n = b.n, i = blockIdx.x, second = blockIdx.y;
    if (i >= n) return;
    const double *m = second ? b.g : b.h, *x = second ? b.h : b.g;
    double a = 0.0;
    for (int p = threadIdx.x + (second && threadIdx.x == 0 ? kTcSumThreads : 0); p < n; p += kTcSumThreads)
        a = fma(m[abs(i - p)], x[p], a);
    a = tc_cta_sum(a);
    if (threadIdx.x != 0) return;
    if (second) b.w[i] = i > 0 ? a + b.h[i] : a;
    else b.wc[i] = tc_add3(a, b.h[i], b.g[i], &b.wc_low[i]);
}

// One CTA per entry i of D's first column, g + wc + G wc.
__global__ void __launch_bounds__(kTcSumThreads) tc_first(const __grid_constant__ TcBuilds all) {
    const TcBuild& b = all.axis[blockIdx.z];
    const int n = b.n, i = blockIdx.x;
    if (i >= n) return;
    double a = 0.0;
    for (int p = threadIdx.x; p < n; p += kTcSumThreads) a = fma(b.g[abs(i - p)], b.wc[p], a);
    a = tc_cta_sum(a);
    if (threadIdx.x == 0) b.d0[i] = tc_add3(a + b.wc_low[i], b.wc[i], b.g[i], &b.d0_low[i]);
}

// The diagonals of D, 32 a CTA. D is symmetric and centrosymmetric (D[i][j] =
// D[n-1-i][n-1-j]): only the first ceil(n/2) rows are formed and stored. Each warp
// walks a quarter of the rows twice, for their sum and then, from the sum of the
// quarters before, for the entries. The FP64 pipe bounds it (a warp alone on its
// scheduler issues one FP64 operation in 64 cycles): the terms of eight rows are
// summed plainly, which are small beside the entry, and only their sum is added with
// compensation. n = 1024, two axes: 215 us with every term compensated by one warp.
__global__ void __launch_bounds__(128) tc_diagonals(const __grid_constant__ TcBuilds all) {
    constexpr int U = 8;
    const TcBuild& b = all.axis[blockIdx.z];
    const int n = b.n, lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int d = blockIdx.x * 32 + lane, half = (n + 1) / 2;
    __shared__ double part[2][3][32];
    const double *g = b.g, *w = b.w;
    const int rows = min(half, n - d);  // of this diagonal; none for d >= n
    const int quarter = (half + 2) / 4, first = 1 + warp * quarter, last = min(rows, first + quarter);
    double* D = b.D;
    auto put = [&](int i, double v) {
        D[(size_t)i * n + i + d] = v;
        if (i + d < half) D[(size_t)(i + d) * n + i] = v;
    };
    auto walk = [&](TcSum& a, bool store) {
        for (int i0 = first; i0 < last; i0 += U) {
            double p = 0.0;
            const double v = a.s + a.c;
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const int i = i0 + q;
                if (i >= last) continue;
                p = fma(2.0 * __ldg(g + i), __ldg(w + i + d), fma(2.0 * __ldg(w + i), __ldg(g + i + d), p));
                if (store) put(i, v + p);
            }
            a.add(p);
        }
    };
    TcSum a;
    if (warp < 3) {
        walk(a, false);
        part[0][warp][lane] = a.s;
        part[1][warp][lane] = a.c;
    }
    __syncthreads();
    if (rows <= 0) return;
    a = TcSum();
    a.s = b.d0[d];
    a.c = b.d0_low[d];
    if (warp == 0) put(0, a.s);
    for (int k = 0; k < warp; ++k) {
        a.add(part[0][k][lane]);
        a.c += part[1][k][lane];
    }
    walk(a, true);
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

__global__ void __launch_bounds__(256) tc_max(const __grid_constant__ TcBuilds all) {
    const TcBuild& b = all.axis[blockIdx.z];
    const int n = b.n, parts = parts_of(n), rows = rows_of(n);
    const double* D = b.D;
    double m = 0.0;
    const int total = parts * rows * rows;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int p = t / (rows * rows), r = t % (rows * rows);
        m = fmax(m, fabs(tc_entry(D, n, parts, rows, p, r / rows, r % rows)));
    }
    for (int w = 16; w > 0; w >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, w));
    if (threadIdx.x % 32 == 0) atomicMax(&b.report->largest, (unsigned long long)__double_as_longlong(m));
}

// Digits of every entry (NS places of B bits), written as 8 KB blocks of 128 rows x
// 32 columns: core matrices of 8 rows x 8 columns, rows first. Order of the
// blocks, the order in which a CTA streams them: (part, 32 columns, place) up to
// 256 points, (128 rows, 32 columns, part, place) above. One CTA per (row,
// part); report as in tc_build.
__global__ void __launch_bounds__(128) tc_digits(const __grid_constant__ TcBuilds all) {
    const TcBuild& b = all.axis[blockIdx.z];
    const int n = b.n, parts = parts_of(n), rows = rows_of(n), kp = kp_of(n), NS = all.slices, B = all.bits;
    const int row = blockIdx.x, p = blockIdx.y, nkc = kp / 32;
    if (p >= parts || row >= (rows + 127) / 128 * 128) return;
    const double* D = b.D;
    __half* img = static_cast<__half*>(b.img);
    TcReport* report = b.report;
    const double m = __longlong_as_double((long long)b.report->largest);
    int f = 0;
    if (m > 0.0) {
        f = ilogb(m) + 1;  // m < 2^f: the top digit has one bit more
        f = f < -200 ? -200 : f;
    }
    if (row == 0 && p == 0 && threadIdx.x == 0) report->scale = f;
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
        // order s takes the row's places 1 .. s - 1, the last of them times the top
        // digit of the line (see TcReport)
        if (threadIdx.x < 10) {
            const int h = threadIdx.x / 5, s = 2 + threadIdx.x % 5;
            int reach = sum[s - 2] << (1 - h);
            for (int j = 0; j < s - 2; ++j) reach += sum[j];
            atomicMax(&report->sums[h][s - 2], reach);
        }
    }
    if (threadIdx.x == 0) atomicMax(&report->row_sum, (int)(total >> 10));
}

}  // namespace

size_t tc_image_bytes(int n, int slices) { return (size_t)parts_of(n) * ((rows_of(n) + 127) / 128) * (kp_of(n) / 32) * slices * 8192; }
size_t tc_scratch_bytes(int n) { return sizeof(double) * ((size_t)((n + 1) / 2) * n + 7 * (size_t)n); }

cudaError_t tc_build(int count, const TcBuildAxis* axes, int slices, int bits, void* scratch, cudaStream_t s) {
    TcBuilds all{};
    all.slices = slices;
    all.bits = bits;
    unsigned char* at = static_cast<unsigned char*>(scratch);
    int n = 0, rows = 0, parts = 1;
    for (int l = 0; l < count; ++l) {
        TcBuild& b = all.axis[l];
        b.n = axes[l].n;
        b.spectra = axes[l].spectra;
        b.img = axes[l].img;
        b.report = axes[l].report;
        double* d = reinterpret_cast<double*>(at);
        double** arrays[7] = {&b.g, &b.h, &b.wc, &b.wc_low, &b.w, &b.d0, &b.d0_low};
        for (double** a : arrays) {
            *a = d;
            d += b.n;
        }
        b.D = d;
        at += tc_scratch_bytes(b.n);
        n = std::max(n, b.n);
        rows = std::max(rows, (rows_of(b.n) + 127) / 128 * 128);
        parts = std::max(parts, parts_of(b.n));
    }
    tc_columns<<<dim3(n / 2 + 1, 2, count), kTcSumThreads, 0, s>>>(all);
    tc_vectors<<<dim3(n, 2, count), kTcSumThreads, 0, s>>>(all);
    tc_first<<<dim3(n, 1, count), kTcSumThreads, 0, s>>>(all);
    tc_diagonals<<<dim3((n + 31) / 32, 1, count), 128, 0, s>>>(all);
    tc_max<<<dim3(std::max(1, std::min(64, n / 4)), 1, count), 256, 0, s>>>(all);
    tc_digits<<<dim3(rows, parts, count), 128, 0, s>>>(all);
    return cudaGetLastError();
}

bool tc_accept(int n, int slices, const void* img, const TcReport& report, TcAxis* ax) {
    ax->n = n;
    ax->parts = parts_of(n);
    ax->rows = rows_of(n);
    ax->kp = kp_of(n);
    ax->scale = report.scale;
    ax->headroom = 0;
    if (slices != kTcSlices) {
        // FP32: the sums are rounded to 24 bits like any FP32 sum. With entries of 1/2
        // and more (long steps: D cancels most of x) the FFT passes are the more
        // accurate ones; a tiny f would leave the exponent range of the closing products.
        if (report.scale > -1 || report.scale < -60) return false;
        ax->img = img;
        return true;
    }
    // Digits of x are at most 2^(B-1) in size, the top one 2^B, or 2^(B-1) too if lines
    // are scaled by one more bit (headroom). The accumulators of orders up to 5 must
    // stay within 2^24 (FP32 holds every integer of that size), order 6 within 2^25 and
    // order 7 anywhere: a unit lost there is below 2^-56 of the line's largest value.
    // The reach of each order is that of one row: added up from the largest sum of each
    // place over all rows it came to 1.25 times as much, and refused 1 in 40 ordinary
    // parameter sets at 1024 points, whose passes then took 205 us instead of 62.
    int headroom = -1;
    for (int h = 0; h < 2 && headroom < 0; ++h) {
        bool ok = true;
        for (int s = 2; s <= 6; ++s)
            ok = ok && std::ldexp((double)report.sums[h][s - 2], kTcBits - 1) <= std::ldexp(1.0, s <= 5 ? 24 : 25);
        if (ok) headroom = h;
    }
    if (headroom < 0) return false;
    // a row's sum of |entries| / 2^f, so that the 64-bit sums of the pass cannot overflow
    if (report.row_sum > 4 << 10 || report.scale > 2) return false;
    ax->headroom = headroom;
    ax->img = img;
    return true;
}

}  // namespace sfac
