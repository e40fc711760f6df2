// sfac_tc_tile.cuh - FP64 lines as exact digit products on the tensor cores.
//
// The linear factor of an axis, P = e^{tau/2 C} e^{tau S} e^{tau/2 C}, is a real
// n x n matrix, and a pass computes y = x + D x, D = P - I, for every line. The
// FP64 pipe of sm_103a does 4 flops a clock per SM, so the six FFTs of a line
// were bound by it (93% busy); the tensor cores do 8192 FP16 flops a clock. D x
// is therefore formed from digits (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication", Numer. Algorithms 59, 2012):
//  - a line is scaled by a power of two above its largest value and rounded to
//    54 fractional bits, cut into six signed digits of 9 bits (FP16 integers);
//    D's entries likewise, once per plan (sfac_tc_build.cu);
//  - the products of digit place i of x with place j of D are summed by
//    tcgen05.mma into one FP32 accumulator per order i + j = 2..7, whole numbers
//    all. Orders 2..5 stay within 2^24, so their sums are exact; order 6 within
//    2^25, and a unit lost there or in order 7 is below 2^-56 of the line's largest
//    value (tc_accept checks the plan's own D); orders from 8 on are left out;
//  - the six sums are added with their weights in 64-bit integers, and
//    y = x + D x is rounded once.
// Against 80-bit arithmetic the increment is within 0.1e-16 to 3e-16 (2-norm,
// relative to the line, for |D| from 0.05 to 2), the FFT passes within 5e-16.
//
// Lines of more than 128 points are folded: D is centrosymmetric (C and S are
// symmetric Toeplitz), so it maps the sums x_k + x_{n-1-k} and the differences
// x_k - x_{n-1-k} each into themselves, two operators of half the size (half the
// products). The operator is the A operand (128 outputs are the M of the MMA),
// the digits of LT lines are the B operand: digit places stacked along N, so
// that one MMA multiplies a digit place of D with up to four places of x and
// writes the orders, neighbouring in tensor memory, in one go. D's digits are
// streamed from L2 in 8 KB blocks through a ring of bulk copies.
//
// Measured (side by side, n = 256, 65536 lines): a pass of six FFTs on the FP64 pipe
// took 1.90 ms (2.15 ms with the flow), this one 0.21 ms (0.27-0.31 ms). What bounds
// it now: the phases of a tile follow each other (barrier stalls 2.2-3.1 per issue), with
// the integer ALU, 64 operations a clock and SM, 38% busy over the whole pass, the
// tensor pipe 18%, L2 10%. Tiles of 32 lines in two CTAs an SM did not overlap them:
// a ring of two blocks each waited for the operator (820 us).
//
// A CTA is THREADS computing threads (one warp of them also issues the
// products) and one more warp that issues the copies of the ring. Both issuing
// loops run on whole warps with uniform control flow and elect a lane for each
// instruction: run by a single thread of a divergent branch they took 460
// cycles a block, four times as long as its products.
#pragma once

#include "sfac_jq_fixed.cuh"
#include "sfac_tc.h"
#include "sfac_tcgen05.cuh"

namespace sfac {

constexpr int kTcOrders = 6;         // accumulated orders 2..7
constexpr unsigned kTcBlock = 8192;  // a streamed block: 128 rows x 32 columns of FP16
constexpr int kTcMaxStages = 24;

// S: digit places (6: FP64, 3: FP32).
template <int PARTS, int LT, int S = kTcSlices>
struct TcShape {
    static constexpr int SLICES = S;
    static constexpr int THREADS = LT >= 64 ? 512 : (LT == 32 ? 256 : 128);
    static constexpr int UPT = LT * 16 / THREADS;       // units (line, 8 columns) a thread holds
    // Digits: bytes between 8-column chunks. Core matrices must stay aligned to
    // their 128 bytes.
    static constexpr int LBO = S * LT * 16;
    static constexpr int PITCH = S == 6 ? LT * 8 + 8 : LT * 4 + 4;  // results: bytes between rows (padded: banks)
    // accumulator columns of a part (LT = 8: a place more, see tc_products)
    static constexpr int REGION = LT == 8 ? (S == 6 ? 8 : 4) * LT : S * LT;
    // A warp of its own for the ring's copies; with 16 computing warps it would
    // cost them a quarter of their registers (128 -> 96), there one of them issues
    // the copies while the others wait for the products.
    static constexpr bool OWN_PRODUCER = THREADS < 512;
    static constexpr int TOTAL = THREADS + (OWN_PRODUCER ? 32 : 0);
    // LT = 64: the accumulators of one part fill tensor memory, the parts run in turn
    static constexpr bool TWO_PHASES = PARTS == 2 && S * PARTS * LT > 512;
    static constexpr int NEED = (TWO_PHASES ? 1 : PARTS) * REGION;
    static constexpr int COLS = NEED <= 64 ? 64 : NEED <= 128 ? 128 : NEED <= 256 ? 256 : 512;
    __host__ __device__ static constexpr int part_bytes(int kp) { return kp / 8 * LBO; }
    // Ring of operator blocks: what shared memory the digits leave, at most 24
    // blocks. Where it is deep enough a stage is three blocks: the waits of either
    // side cost about 200 cycles a stage, more than one block's products.
    static constexpr int CTAS = S == 6 || LT >= 64 ? 1 : 2;  // resident CTAs an SM
    static constexpr int RING_OFFSET = PARTS * part_bytes(128);
    static constexpr int FIT = (231000 / CTAS - 2000 * (CTAS - 1) - RING_OFFSET) / (int)kTcBlock;
    static constexpr int G = FIT >= 9 ? 3 : 1;  // blocks of a stage
    static constexpr int STAGES = (FIT < kTcMaxStages ? FIT : kTcMaxStages) / G;
    static constexpr int SMEM = RING_OFFSET + STAGES * G * (int)kTcBlock;
};

// One pass over lines: element k of line L sits at
// (L / inner) * n * inner + L % inner + k * inner.
template <typename R>
struct TcPassT {
    const R* src;
    R* dst;
    long long inner, lines, ntiles;
    int n, rows, kp, scale, headroom;
    int prefetch;  // lines in device memory: later tiles may be prefetched
    int jq_in, jq_out;
    JqFixed jin, jout;
};

using TcPass = TcPassT<double>;

template <typename R>
inline TcPassT<R> tc_pass_of(const TcAxis& ax, const PassArgs& a) {
    TcPassT<R> p;
    p.src = static_cast<const R*>(a.u);
    p.dst = static_cast<R*>(a.u) + a.out_shift;
    p.inner = a.inner;
    p.lines = a.outer * a.inner;
    p.ntiles = 0;
    p.n = ax.n;
    p.rows = ax.rows;
    p.kp = ax.kp;
    p.scale = ax.scale;
    p.headroom = ax.headroom;
    p.prefetch = !a.host_io;
    p.jq_in = a.jq_in;
    p.jq_out = a.jq_out;
    p.jin = make_jq_fixed(a.jq_in_E, a.jq_in_1mE);
    p.jout = make_jq_fixed(a.jq_out_E, a.jq_out_1mE);
    return p;
}

// Barriers and flags of a CTA, in shared memory.
struct TcShared {
    uint64_t full[kTcMaxStages], empty[kTcMaxStages], done, never;
    uint32_t tmem;
    int abort;
};

// Ring and barrier positions of a CTA's warps; every lane of a warp holds the
// same values. The warp that issues the copies keeps its own ring position, the
// next stage of the image, and how many stages are still to come.
struct TcState {
    int stage = 0;
    unsigned parity = 0;       // consumer: of full; producer: of empty (starts at 1)
    unsigned done_parity = 0;
    int block = 0;
    long long left = 0;
};

__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// Waits on `bar` with the whole (converged) warp, at most `limit` cycles; a wait
// that runs out, or that sees another warp's that did, returns false. NAP: polls
// seldom (the producer: its polls took issue slots from the other warps).
template <bool NAP = false>
__device__ __forceinline__ bool tc_wait(uint64_t* bar, unsigned parity, long long limit, int* abort) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    for (;;) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        const bool late = clock64() - t0 > limit;
        if (__any_sync(0xffffffffu, late || *reinterpret_cast<volatile int*>(abort) != 0)) {
            *reinterpret_cast<volatile int*>(abort) = 1;
            return false;
        }
        if (NAP) __nanosleep(100);
    }
}

// Barrier 1 among the NT computing threads; the second form also ANDs a flag.
template <int NT>
__device__ __forceinline__ void tc_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}
template <int NT>
__device__ __forceinline__ bool tc_sync_and(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(NT)
        : "memory");
    return r != 0;
}

constexpr unsigned long long kTcBias = [] {
    unsigned long long b = 0;
    for (int i = 0; i < kTcSlices; ++i) b += 1ULL << (kTcBits * i + kTcBits - 1);
    return b + (1ULL << (kTcBits * kTcSlices - 1));  // the top digit has one bit more
}();

// A value of a line whose largest one has the exponent field E, in units of
// 2^(E - 1082): at most 2^60, the grid far below the FP64 rounding of the
// line's largest values.
__device__ __forceinline__ long long tc_fixed(double v, int E) {
    const int hi = __double2hiint(v);
    const int ex = (hi >> 20) & 0x7ff;
    const unsigned mh = (hi & 0xfffff) | (ex ? 0x100000u : 0u);
    const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(v)) << 7;
    int sh = E - (ex ? ex : 1);
    sh = sh > 63 ? 63 : sh;
    const long long f = (long long)(m >> sh);
    return hi < 0 ? -f : f;
}

// Exponent field of a line's scale, from its largest value's field Eb (0: zero or
// subnormal values).
__device__ __forceinline__ int tc_scale_of(int Eb, int headroom) { return max(Eb, 1) + headroom; }
// Whether every result of the line is zero or a normal number.
__device__ __forceinline__ bool tc_plain(int Eb) { return (unsigned)(Eb - 61) <= 2041u - 61u; }

// Back to FP64, rounded to nearest (ties away), in a plain line: |y| < 2^63.
__device__ __forceinline__ double tc_to_double(long long y, int E) {
    if (y == 0) return 0.0;
    const unsigned long long m = y < 0 ? 0ULL - (unsigned long long)y : (unsigned long long)y;
    const int lz = __clzll((long long)m);
    const unsigned long long t = (((m << lz) >> 10) + 1) >> 1;  // 2^52 .. 2^53
    const int e = E + 3 - lz;                                   // exponent field less one
    const long long bits = (long long)t + ((long long)e << 52);
    return __longlong_as_double(bits | (y & (long long)0x8000000000000000ULL));
}
// The same in any line: subnormal results, infinities, and NaN throughout a line
// that holds an infinity or a NaN (Eb = 2047).
__device__ __forceinline__ double tc_to_double_any(long long y, int E, int Eb) {
    if (Eb == 2047) return __longlong_as_double(0x7ff8000000000000LL);
    if (y == 0) return 0.0;
    const unsigned long long m = y < 0 ? 0ULL - (unsigned long long)y : (unsigned long long)y;
    const int lz = __clzll((long long)m);
    const int e = E + 3 - lz;
    long long bits;
    if (e >= 2046)
        bits = 0x7ff0000000000000LL;
    else if (e >= 0)
        bits = (long long)((((m << lz) >> 10) + 1) >> 1) + ((long long)e << 52);
    else  // in units of 2^-1074; y is in units of 2^(E - 1082)
        bits = (long long)(E >= 8 ? m << (E - 8) : (m + (1ULL << (7 - E))) >> (8 - E));
    return __longlong_as_double(bits | (y & (long long)0x8000000000000000ULL));
}

// V sums (as bits) back to FP64; Eb(r): the largest field of value r's line,
// cell(r): a shared-memory word that is this thread's own. The rare lines go through
// one rolled loop in shared memory (a 3D 63^3 step 138.0 -> 139.6 us): unrolled
// beside the plain code, or with the values picked out of registers, they took
// 141 us, as the code of a pass of one round is fetched for one use.
template <int V, typename F, typename C>
__device__ __forceinline__ void tc_to_doubles(double (&x)[V], int headroom, F Eb, C cell) {
    bool plain = true;
#pragma unroll
    for (int r = 0; r < V; ++r) plain = plain && tc_plain(Eb(r));
    if (__builtin_expect(plain, 1)) {
#pragma unroll
        for (int r = 0; r < V; ++r) x[r] = tc_to_double(__double_as_longlong(x[r]), tc_scale_of(Eb(r), headroom));
    } else {
#pragma unroll
        for (int r = 0; r < V; ++r) *cell(r) = x[r];
#pragma unroll 1
        for (int r = 0; r < V; ++r) {
            double* p = cell(r);
            *p = tc_to_double_any(__double_as_longlong(*p), tc_scale_of(Eb(r), headroom), Eb(r));
        }
#pragma unroll
        for (int r = 0; r < V; ++r) x[r] = *cell(r);
    }
}

// Digit place q (0: most significant) of two biased values whose lowest digit is at
// bit SB, as two FP16 integers.
template <int SB>
__device__ __forceinline__ uint32_t tc_digit_pair(unsigned long long f0, unsigned long long f1, int q) {
    const int sh = SB + kTcBits * (kTcSlices - 1 - q);
    const unsigned mask = q == 0 ? 0x7ffu : 0x1ffu;
    const unsigned short off = q == 0 ? 0x6600 : 0x6500;  // 1024 + 512, 1024 + 256
    const unsigned a = (unsigned)(f0 >> sh) & mask, b = (unsigned)(f1 >> sh) & mask;
    const unsigned h = (a | (b << 16)) + 0x64006400u;  // 1024 + field, twice
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(off)));
    return *reinterpret_cast<const uint32_t*>(&d);
}

// The eight biased values F[0..7] of one line and chunk -> six FP16 digits each,
// stored as 16-byte rows of the B operand (row = place * LT + line).
template <int LT, int SB>
__device__ __forceinline__ void tc_put_digits(unsigned char* chunk, int line, const unsigned long long (&F)[8]) {
#pragma unroll
    for (int q = 0; q < kTcSlices; ++q) {
        const int r = q * LT + line;
        *reinterpret_cast<uint4*>(chunk + (r >> 3) * 128 + (r & 7) * 16) =
            make_uint4(tc_digit_pair<SB>(F[0], F[1], q), tc_digit_pair<SB>(F[2], F[3], q),
                       tc_digit_pair<SB>(F[4], F[5], q), tc_digit_pair<SB>(F[6], F[7], q));
    }
}

// A sum in units of 2^(E - 1082 + f) in units of 2^(E - 1082), rounded.
__device__ __forceinline__ long long tc_align(long long v, int f) {
    if (f >= 0) return v << f;
    if (f > -32) {  // a funnel shift; f is the same for the whole launch
        const unsigned long long t = (unsigned long long)(v + (1LL << (-f - 1)));
        return (long long)(((unsigned long long)(unsigned)((int)(t >> 32) >> -f) << 32) |
                           __funnelshift_r((unsigned)t, (unsigned)(t >> 32), (unsigned)-f));
    }
    const int right = min(-f, 62);
    return (v + (1LL << (right - 1))) >> right;
}

// The order sums of one output -> the 64-bit integer sum in units of 2^-6 of
// order 6.
__device__ __forceinline__ long long tc_combine(const float (&a)[kTcOrders]) {
    const long long hi = (long long)__float2int_rn(a[0]) * (1 << 18) + (long long)__float2int_rn(a[1]) * (1 << 9) +
                         __float2int_rn(a[2]);
    const int r = __float2int_rn(a[5] * 0.125f);
    const long long lo = (long long)__float2int_rn(a[3]) * (1 << 15) + (long long)__float2int_rn(a[4]) * 64 + r;
    return (hi << 24) + lo;
}

// 32 aligned bytes, one sector of L2, a lane.
__device__ __forceinline__ void ld_sector(const double* p, double (&v)[4]) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st_sector(double* p, double a, double b, double c, double d) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
}

// Eight consecutive values at any 8-byte aligned p: the aligned sectors around
// them, then a shift. Narrower loads, each lane in sectors of its own, come back to a
// sector that has left the small L1 beside the tile (16-byte loads: a contiguous
// pass of 256^3 took 227 us, a strided one 208). `inside`: the sectors around the
// values lie in the field (tc_groups_inside).
__device__ __forceinline__ void tc_load8(const double* p, bool inside, double (&v)[8]) {
    const unsigned s = (unsigned)(reinterpret_cast<uintptr_t>(p) >> 3) & 3u;
    if (s == 0) {
        double t[4];
        ld_sector(p, t);
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = t[r];
        ld_sector(p + 4, t);
#pragma unroll
        for (int r = 0; r < 4; ++r) v[4 + r] = t[r];
        return;
    }
    if (!inside) {
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = p[r];
        return;
    }
    double t[12], h[11];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double w[4];
        ld_sector(p - s + 4 * i, w);
#pragma unroll
        for (int r = 0; r < 4; ++r) t[4 * i + r] = w[r];
    }
#pragma unroll
    for (int r = 0; r < 11; ++r) h[r] = s & 1u ? t[r + 1] : t[r];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = s & 2u ? h[r + 2] : h[r];
}
__device__ __forceinline__ void tc_store8(double* p, const double (&v)[8]) {
    auto two = [&](int i) { *reinterpret_cast<double2*>(p + i) = make_double2(v[i], v[i + 1]); };
    auto four = [&](int i) { st_sector(p + i, v[i], v[i + 1], v[i + 2], v[i + 3]); };
    switch ((unsigned)(reinterpret_cast<uintptr_t>(p) >> 3) & 3u) {
        case 0: four(0), four(4); break;
        case 1: p[0] = v[0], two(1), four(3), p[7] = v[7]; break;
        case 2: two(0), four(2), two(6); break;
        default: p[0] = v[0], four(1), two(5), p[7] = v[7]; break;
    }
}

// Asks L2 for the lines of a later tile, 128 bytes a lane (threads `me` of
// `many`): their loads then wait for L2 and not for memory.
template <int LT, bool STRIDED, typename R>
__device__ __forceinline__ void tc_prefetch(const TcPassT<R>& g, long long tile, int me, int many) {
    constexpr int PER = 128 / (int)sizeof(R);  // values of 128 bytes
    if (!g.prefetch || tile >= g.ntiles) return;
    if constexpr (STRIDED) {
        constexpr int PIECES = LT / PER > 0 ? LT / PER : 1;
        const long long L = tile * LT + me % PIECES * PER;
        if (L >= g.lines) return;
        const long long o = L / g.inner;
        const R* p = g.src + o * g.n * g.inner + (L - o * g.inner);
        for (int k = me / PIECES; k < g.n; k += many / PIECES)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p + k * g.inner));
    } else {
        const long long first = tile * LT * g.n, last = min((tile + 1) * LT, g.lines) * g.n;
        for (long long i = first + me * PER; i < last; i += many * PER)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(g.src + i));
    }
}

// The producer: up to `count` more stages of an image of `stages` of them (st.left
// counts stages too). Before stage number `early` of these it waits for the
// previous pass: the first ring needs no room, but the room for more comes only
// once the lines are loaded, and the limit of that wait must not run while the
// previous pass does (a 4096 x 200 step under a limit of 100 us gave up).
template <int STAGES, int G>
__device__ __forceinline__ bool tc_produce(TcShared& sh, TcState& st, unsigned char* ring, const unsigned char* img,
                                           int stages, long long count, long long limit, long long early = -1) {
    constexpr unsigned BYTES = G * kTcBlock;
    if (count > st.left) count = st.left;
#pragma unroll 1
    for (long long c = 0; c < count; ++c) {
        if (c == early) pass_wait_for_previous();
        if (!tc_wait<true>(&sh.empty[st.stage], st.parity, limit, &sh.abort)) return false;
        if (elect_one()) {
            mbar_expect_tx(&sh.full[st.stage], BYTES);
            bulk_load(ring + st.stage * BYTES, img + (size_t)st.block * BYTES, BYTES, &sh.full[st.stage]);
        }
        __syncwarp();
        --st.left;
        if (++st.block == stages) st.block = 0;
        if (++st.stage == STAGES) {
            st.stage = 0;
            st.parity ^= 1u;
        }
    }
    return true;
}

// The products of parts [part0, part1), issued by one whole warp; they arrive on
// sh.done. A block holds one digit place J of D for 32 columns; it meets the
// places 1 .. S + 1 - J of x (orders J + 1 .. S + 1). One compact loop: unrolled over the
// places, a narrow tile spent most of the time fetching instructions.
template <int PARTS, int LT, int STAGES, int G, int S = kTcSlices>
__device__ __forceinline__ void tc_products(TcShared& sh, TcState& st, unsigned char* digits, unsigned char* ring,
                                            uint32_t tmem, int part0, int part1, int kp, long long limit) {
    using Sh = TcShape<PARTS, LT, S>;
    const uint64_t a0 = tc_desc(smem_u32(ring), 2048, 128), b0 = tc_desc(smem_u32(digits), Sh::LBO, 128);
    const int stages = (kp >> 5) * S / G;
    bool ok = true;
#pragma unroll 1
    for (int part = part0; ok && part < part1; ++part) {
        const uint32_t d0 = tmem + (Sh::TWO_PHASES ? 0 : part * Sh::REGION);
        uint64_t bd = b0 + (uint32_t)(part * Sh::part_bytes(kp) >> 4);
        int j = 0;  // J - 1
        uint32_t later = 0;
#pragma unroll 1
        for (int b = 0; b < stages; ++b) {
            ok = tc_wait(&sh.full[st.stage], st.parity, limit, &sh.abort);
            if (!ok) break;
            uint64_t ad = a0 + (uint32_t)(st.stage * (G * kTcBlock >> 4));
#pragma unroll 1
            for (int q = 0; q < G; ++q, ad += kTcBlock >> 4) {
                const int m = S - j;
                // N is a multiple of 16 (LT = 8: an even number of places, whose last may
                // go to an unused order) and at most 256 (LT = 64: 4 places, then the rest)
                const int w = S * LT > 256 ? min(m, 4) : (LT == 8 ? (m + 1) & ~1 : m);
                const uint32_t d = d0 + j * LT;
                const uint32_t idesc = tc_idesc_f16(128, 0) + ((uint32_t)(w * LT) >> 3 << 17);
                // place 1 reaches every order: its first products overwrite them
                const uint32_t acc = j == 0 ? later : 1u;
                if (elect_one()) {
                    tc_mma_f16(d, ad, bd, idesc, acc);
                    if (S * LT > 256 && m > 4)
                        tc_mma_f16(d + 4 * LT, ad, bd + (4 * LT * 16 >> 4),
                                   tc_idesc_f16(128, 0) + ((uint32_t)((m - 4) * LT) >> 3 << 17), acc);
                    tc_mma_f16(d, ad + (4096 >> 4), bd + (2 * Sh::LBO >> 4), idesc, 1u);
                    if (S * LT > 256 && m > 4)
                        tc_mma_f16(d + 4 * LT, ad + (4096 >> 4), bd + (2 * Sh::LBO >> 4) + (4 * LT * 16 >> 4),
                                   tc_idesc_f16(128, 0) + ((uint32_t)((m - 4) * LT) >> 3 << 17), 1u);
                    if (q == G - 1) tc_commit(&sh.empty[st.stage]);
                }
                __syncwarp();
                if (++j == S) {
                    j = 0;
                    later = 1;
                    bd += 4 * Sh::LBO >> 4;
                }
            }
            if (++st.stage == STAGES) {
                st.stage = 0;
                st.parity ^= 1u;
            }
        }
    }
    if (elect_one()) tc_commit(&sh.done);
    __syncwarp();
}

// Line L's first element (an index), with a 32-bit division where it suffices.
__device__ __forceinline__ long long tc_line_base(long long L, long long inner, int n) {
    if (((L | inner) >> 32) == 0) {
        const unsigned o = (unsigned)L / (unsigned)inner;
        return (long long)o * n * inner + ((unsigned)L - o * (unsigned)inner);
    }
    const long long o = L / inner;
    return o * n * inner + (L - o * inner);
}

// The CTA's tiles of LT lines, by the computing threads: false if a wait ran out.
// smem: the digits (then the results); smax: LT words.
//
// What a tile's 58,000 cycles (n = 256, 64 lines) were spent on, one after the
// other: load 8,500, digits 9,500, products 9,000 and 9,000, sums 4,500 and
// 4,500, update and store 12,500. Two of these overlap others: the digits of the
// odd part are written while the even part's products run, and a unit's next
// values are loaded into its registers as soon as it is stored.
template <int PARTS, int LT, bool STRIDED, int STAGES>
__device__ __forceinline__ bool tc_tiles(const TcPass& g, unsigned char* smem, unsigned char* ring, unsigned* smax,
                                         TcShared& sh, TcState& st, uint32_t tmem, const unsigned char* img, int tid,
                                         long long limit) {
    using Sh = TcShape<PARTS, LT>;
    constexpr int NT = Sh::THREADS, UPT = Sh::UPT, LBO = Sh::LBO;
    constexpr int VPU = PARTS == 2 ? 16 : 8;  // values of a unit
    constexpr bool TWO_PHASES = Sh::TWO_PHASES;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n = g.n, rows = g.rows, kp = g.kp, nch = kp >> 3;
    const int part_bytes = Sh::part_bytes(kp);

    // Units (line, chunk c of 8 columns, and their mirror images). Strided axis:
    // lanes along the lines; contiguous axis: a warp takes 4 chunks (256 bytes) of
    // 8 lines.
    double x[UPT][VPU];  // then, as integers, the fixed-point values
    int uline[UPT] = {}, uc[UPT] = {};
    auto load = [&](int it, long long tile) {
        const int c = uc[it];
        const long long L = tile * LT + uline[it];
#pragma unroll
        for (int r = 0; r < VPU; ++r) x[it][r] = 0.0;
        if (uline[it] < 0 || L >= g.lines) return;
        const double* p = g.src + (STRIDED ? tc_line_base(L, g.inner, n) : L * n);
        if (!STRIDED && 8 * c + 8 <= rows) {
            double v[8];
            tc_load8(p + 8 * c, tc_groups_inside(L * n + 8 * c, g.lines * n), v);
#pragma unroll
            for (int r = 0; r < 8; ++r) x[it][r] = v[r];
            if constexpr (PARTS == 2) {
                tc_load8(p + n - 8 - 8 * c, tc_groups_inside(L * n + n - 8 - 8 * c, g.lines * n), v);
#pragma unroll
                for (int r = 0; r < 8; ++r) x[it][8 + r] = v[7 - r];
            }
            return;
        }
        const long long stride = STRIDED ? g.inner : 1;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int k = 8 * c + r;
            if (k < rows) {
                x[it][r] = p[k * stride];
                if constexpr (PARTS == 2) x[it][8 + r] = p[(n - 1 - k) * stride];
            }
        }
    };
    // digits of one part of a unit: sums and differences in units of 2^(E - 1075),
    // values themselves in units of 2^(E - 1076): at most 2^54 in size, rounded
    auto digits = [&](int it, int part) {
        constexpr int SB = PARTS == 2 ? 7 : 6;
        constexpr unsigned long long bias = (kTcBias << SB) + (1ULL << (SB - 1));
        if (uline[it] < 0) return;
        unsigned long long F[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            F[r] = bias + __double_as_longlong(x[it][r]);
            if constexpr (PARTS == 2) {
                const long long y = __double_as_longlong(x[it][8 + r]);
                F[r] += part == 0 ? y : -y;
            }
        }
        tc_put_digits<LT, SB>(smem + part * part_bytes + uc[it] * LBO, uline[it], F);
    };
#pragma unroll
    for (int it = 0; it < UPT; ++it) {
        const int u = tid + it * NT;
        uc[it] = STRIDED ? u / LT : (u / 32) / (LT / 8) * 4 + ((u >> 3) & 3);
        uline[it] = uc[it] >= nch ? -1 : STRIDED ? u % LT : (u / 32) % (LT / 8) * 8 + (u & 7);
        load(it, blockIdx.x);
    }

#pragma unroll 1
    for (long long tile = blockIdx.x; tile < g.ntiles; tile += gridDim.x) {
        for (int i = tid; i < LT; i += NT) smax[i] = 0;
        tc_sync<NT>();
#pragma unroll
        for (int it = 0; it < UPT; ++it) {
            if (g.jq_in) jq_flow_fixed_all(x[it], g.jin);
            unsigned m = 0;
#pragma unroll
            for (int r = 0; r < VPU; ++r) m = max(m, (unsigned)__double2hiint(x[it][r]) & 0x7fffffffu);
            if (uline[it] >= 0) atomicMax(&smax[uline[it]], m);
        }
        tc_sync<NT>();
        // ---- digits (two phases: the odd part's by the issuing warps only, see below) ----
        const bool issues = warp < 2;
#pragma unroll
        for (int it = 0; it < UPT; ++it) {
            const int E = tc_scale_of((int)(smax[max(uline[it], 0)] >> 20), g.headroom);
#pragma unroll
            for (int r = 0; r < VPU; ++r) x[it][r] = __longlong_as_double(tc_fixed(x[it][r], E));
            digits(it, 0);
            if (PARTS == 2 && (!TWO_PHASES || issues)) digits(it, 1);
        }
        fence_proxy_async_smem();
        tc_sync<NT>();
#pragma unroll 1
        for (int ph = 0; ph < (TWO_PHASES ? 2 : 1); ++ph) {
            // ---- products: the other warps wait at the barrier, not polling ----
            bool ok = true;
            if (warp == 0) {
                tc_fence_after_sync();
                tc_products<PARTS, LT, STAGES, Sh::G>(sh, st, smem, ring, tmem, TWO_PHASES ? ph : 0, TWO_PHASES ? ph + 1 : PARTS,
                                               kp, limit);
                ok = tc_wait(&sh.done, st.done_parity, limit, &sh.abort);
            }
            if (ph == 0 && !issues) {
                if constexpr (TWO_PHASES) {
#pragma unroll
                    for (int it = 0; it < UPT; ++it) digits(it, 1);
                    fence_proxy_async_smem();
                }
                tc_prefetch<LT, STRIDED>(g, tile + gridDim.x, tid - 64, NT - 64);
            }
            if (!Sh::OWN_PRODUCER && warp == 1)
                tc_produce<STAGES, Sh::G>(sh, st, ring, img, PARTS * (kp >> 5) * kTcSlices / Sh::G,
                                          (TWO_PHASES ? 1 : PARTS) * (kp >> 5) * kTcSlices / Sh::G, limit);
            st.done_parity ^= 1u;
            if (!tc_sync_and<NT>(ok && *reinterpret_cast<volatile int*>(&sh.abort) == 0)) return false;
            tc_fence_after_sync();
            // ---- the order sums -> integers, through shared memory (row, line) ----
            {
                constexpr int GROUPS = NT / 128, CPG = LT / GROUPS < 4 ? 4 : LT / GROUPS;
                const int row = (warp & 3) * 32 + lane;
                const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
                const int col0 = (warp >> 2) * CPG;
                unsigned char* r0 = smem + row * Sh::PITCH;
                unsigned char* r1 = smem + part_bytes + row * Sh::PITCH;
#pragma unroll 1
                for (int cc = col0; cc < col0 + CPG; cc += 4) {
                    __syncwarp();
                    uint32_t t[kTcOrders][4];
#pragma unroll
                    for (int s = 0; s < kTcOrders; ++s) tmem_ld4(taddr + s * LT + cc, t[s]);
                    tc_wait_ld();
                    long long v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float f[kTcOrders];
#pragma unroll
                        for (int s = 0; s < kTcOrders; ++s) f[s] = __uint_as_float(t[s][q]);
                        v[q] = tc_combine(f);
                    }
                    long long w[4];
                    if constexpr (PARTS == 2 && !TWO_PHASES) {
#pragma unroll
                        for (int s = 0; s < kTcOrders; ++s) tmem_ld4(taddr + Sh::REGION + s * LT + cc, t[s]);
                        tc_wait_ld();
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float f[kTcOrders];
#pragma unroll
                            for (int s = 0; s < kTcOrders; ++s) f[s] = __uint_as_float(t[s][q]);
                            w[q] = tc_combine(f);
                        }
                    }
                    if (row < kp) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int off = (cc + q) * 8;
                            long long* p0 = reinterpret_cast<long long*>(r0 + off);
                            long long* p1 = reinterpret_cast<long long*>(r1 + off);
                            if constexpr (PARTS == 1) {
                                *p0 = v[q];
                            } else if constexpr (TWO_PHASES) {
                                if (ph == 0) {
                                    *p0 = v[q];
                                } else {
                                    const long long e = *p0;
                                    *p0 = e + v[q];
                                    *p1 = e - v[q];
                                }
                            } else {
                                *p0 = v[q] + w[q];
                                *p1 = v[q] - w[q];
                            }
                        }
                    }
                }
            }
            tc_fence_before_sync();
            tc_sync<NT>();
        }
        // ---- y = x + D x, the closing flow, store; load the unit's next values ----
#pragma unroll
        for (int it = 0; it < UPT; ++it) {
            const int line = uline[it], c = uc[it];
            const long long L = tile * LT + line;
            if (line >= 0 && L < g.lines) {
                const int Eb = (int)(smax[line] >> 20);
                auto cell = [&](int r) {
                    return reinterpret_cast<double*>(smem + (8 * c + (r & 7)) * Sh::PITCH + line * 8 +
                                                     (r >> 3) * part_bytes);
                };
#pragma unroll
                for (int r = 0; r < VPU; ++r) {
                    const long long v = __double_as_longlong(*cell(r));
                    x[it][r] = __longlong_as_double(__double_as_longlong(x[it][r]) + tc_align(v, g.scale));
                }
                tc_to_doubles(x[it], g.headroom, [=](int) { return Eb; }, cell);
                if (g.jq_out) jq_flow_fixed_all(x[it], g.jout);
                double* p = g.dst + (STRIDED ? tc_line_base(L, g.inner, n) : L * n);
                if (!STRIDED && 8 * c + 8 <= rows) {
                    double v[8];
#pragma unroll
                    for (int r = 0; r < 8; ++r) v[r] = x[it][r];
                    tc_store8(p + 8 * c, v);
                    if constexpr (PARTS == 2) {
#pragma unroll
                        for (int r = 0; r < 8; ++r) v[r] = x[it][15 - r];
                        tc_store8(p + n - 8 - 8 * c, v);
                    }
                } else {
                    const long long stride = STRIDED ? g.inner : 1;
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const int k = 8 * c + r;
                        if (k < rows) {
                            p[k * stride] = x[it][r];
                            if constexpr (PARTS == 2) p[(n - 1 - k) * stride] = x[it][8 + r];
                        }
                    }
                }
            }
            if (tile + gridDim.x < g.ntiles) load(it, tile + gridDim.x);
        }
        tc_sync<NT>();  // results and smax are rewritten by the next tile
    }
    return true;
}

// Sets up a CTA: tensor memory (warp 0), barriers. All threads of the CTA.
template <int COLS, int STAGES>
__device__ __forceinline__ uint32_t tc_setup(TcShared& sh) {
    if (threadIdx.x < 32) tmem_alloc(&sh.tmem, COLS);
    if (threadIdx.x == 32) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&sh.full[i], 1);
            mbar_init(&sh.empty[i], 1);
        }
        mbar_init(&sh.done, 1);
        mbar_init(&sh.never, 1);
        sh.abort = 0;
        fence_mbar_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    return sh.tmem;
}

// A wait of the CTA ran out: before it leaves, its copies and products in flight
// finish (waits bounded again) and the timeout is recorded. `st` of the producer
// warp: the last copy of a stage is the one before the stage's next use.
template <int STAGES>
__device__ __forceinline__ void tc_drain_copies(TcShared& sh, const TcState& st, long long limit) {
    for (int i = 0; i < STAGES; ++i)
        mbar_wait_bounded(&sh.full[i], i < st.stage ? st.parity ^ 1u : st.parity, limit);
}

}  // namespace sfac
