// sfac_jq_fixed.cuh - the nonlinear flow J^Q in FP64 precision on the integer pipe.
//
// J^Q_s(v) = v / sqrt(E + (1 - E) v^2). In FP64 that is about nine operations of
// the FP64 pipe a value (half a cycle of a whole SM each on sm_103a); the tensor-core
// passes leave that pipe idle otherwise, and the flow then took most of their
// time (n = 256: 76,000 of 160,000 cycles a tile of 64 lines). In 64-bit fixed
// point it takes about 65 integer operations, which the SM does 64 of a cycle.
// Error: at most 1.9 units in the last place, 0.25 in the mean (products truncated
// by up to two units of 2^-56). 3D 256^3, the flow's share of a pass: FP64 pipe 245 us, with
// exact 64-bit products 90 us, as it stands 75 us.
#pragma once

#include "sfac_pass.cuh"

namespace sfac {

// Constants of one flow: 1 - E in units of 2^-64, E in units of 2^-60, and both as
// doubles for the values outside the fixed-point range.
struct JqFixed {
    double E, omE;
    unsigned long long om64, E60;
    int fixed;  // E >= 1/4: below, s could lose its leading bits
};

inline __host__ __device__ JqFixed make_jq_fixed(double E, double omE) {
    JqFixed c;
    c.E = E;
    c.omE = omE;
    c.fixed = E >= 0.25 && omE >= 0.0 && omE <= 0.75;
    c.om64 = c.fixed ? (unsigned long long)(omE * 18446744073709551616.0) : 0;
    c.E60 = c.fixed ? (unsigned long long)(E * 1152921504606846976.0) : 0;
    return c;
}

// Whether v has the fixed-point form (not: zero, below 2^-1018, |v| >= 4,
// infinities, NaN; large time steps).
__device__ __forceinline__ bool jq_in_range(double v, const JqFixed& q) {
    const int ex = (__double2hiint(v) >> 20) & 0x7ff;
    return q.fixed && (unsigned)(ex - 5) < 1020u;
}
__device__ __forceinline__ double jq_out_of_range(double v, const JqFixed& q) {
    return v == 0.0 ? v : jq_flow(v, q.E, q.omE);
}

// The upper half of a 64 x 64-bit product, at most 2 units below it: without the
// product of the lower halves and the carry of the other parts' lower words
// (three multiplies and two adds instead of ten instructions).
__device__ __forceinline__ unsigned long long mul_hi_about(unsigned long long a, unsigned long long b) {
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
    return (unsigned long long)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

// The fixed-point form; any value may be passed, the result holds for those in range.
__device__ __forceinline__ double jq_fixed_body(double v, const JqFixed& q) {
    const int hi = __double2hiint(v);
    const int ex = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);  // 53 bits
    // |v| (below 4) in units of 2^-62, v^2 and s = E + (1 - E) v^2 < 16 in units of 2^-60
    const unsigned long long a = (m << 11) >> min(max(1024 - ex, 0), 63);
    const unsigned long long w = mul_hi_about(a, a);
    const unsigned long long s = q.E60 + mul_hi_about(w, q.om64);
    // y0 ~ s^-1/2 from the FP32 unit, in units of 2^-30 (y0 <= 2)
    float y0;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(__uint2float_rn((unsigned)(s >> 32)) * 0x1p-28f));
    const unsigned Y = __float2uint_rn(y0 * 0x1p30f);
    // e = 1 - s y0^2 (below 2^-21 in size), in units of 2^-56
    const long long e = (1LL << 56) - (long long)mul_hi_about(s, (unsigned long long)Y * Y);
    // y = y0 (1 + c), c = e/2 + 3 e^2/8; the next term is below 2^-63
    const int e32 = (int)(e >> 5);
    const long long c = (e >> 1) + ((__mulhi(e32, e32) * 3) >> 17);
    // y in units of 2^-62
    const unsigned long long g = ((unsigned long long)Y << 32) +
                                 (unsigned long long)(((c >> 32) * (long long)Y) << 8) +
                                 (((c & 0xffffffffLL) * (unsigned long long)Y) >> 24);
    // |v| y: 64-bit mantissa product (units of 2^-61 of v's power of two), rounded to 53 bits
    const unsigned long long r = mul_hi_about(m << 11, g);  // 2^59 .. 2^63
    const int lz = __clz((int)(r >> 32)), down = 11 - lz;    // 7 .. 10
    const unsigned long long t = r + (1ULL << 10 >> lz);
    const unsigned lo = __funnelshift_r((unsigned)t, (unsigned)(t >> 32), down);
    const unsigned up = (unsigned)(t >> 32) >> down;
    return __hiloint2double((int)((up + ((unsigned)(ex - lz + 1) << 20)) | ((unsigned)hi & 0x80000000u)), (int)lo);
}

__device__ __forceinline__ double jq_flow_fixed(double v, const JqFixed& q) {
    return jq_in_range(v, q) ? jq_fixed_body(v, q) : jq_out_of_range(v, q);
}

// V values: the fixed-point forms first, without branches between them (their
// long chains of dependent operations overlap), then the values out of range.
template <int V>
__device__ __forceinline__ void jq_flow_fixed_all(double (&x)[V], const JqFixed& q) {
    unsigned rare = 0;
#pragma unroll
    for (int r = 0; r < V; ++r) {
        const bool in = jq_in_range(x[r], q);
        if (!in && x[r] != 0.0) rare |= 1u << r;
        x[r] = in ? jq_fixed_body(x[r], q) : x[r];
    }
    if (rare) {
#pragma unroll 1
        for (int r = 0; r < V; ++r) {
            if (!((rare >> r) & 1u)) continue;
#pragma unroll
            for (int s = 0; s < V; ++s)
                if (s == r) x[s] = jq_out_of_range(x[s], q);
        }
    }
}

}  // namespace sfac
