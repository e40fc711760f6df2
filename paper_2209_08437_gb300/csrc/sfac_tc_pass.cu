// sfac_tc_pass.cu - the FP64 axis pass as exact digit products on the tensor cores.
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
//    tcgen05.mma into one FP32 accumulator per order i + j = 2..7. All of them
//    are whole numbers of at most 2^24, so every sum is exact (tc_accept checks
//    the bound for the plan's own D); orders from 8 on are left out;
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
#include <atomic>

#include "sfac_jq_fixed.cuh"
#include "sfac_tc.h"
#include "sfac_tcgen05.cuh"

namespace sfac {
namespace {

constexpr int NS = kTcSlices, DB = kTcBits;
constexpr int kOrders = 6;        // accumulated orders 2..7
constexpr unsigned kBlock = 8192;  // a streamed block: 128 rows x 32 columns of FP16
constexpr unsigned long long kBias = [] {
    unsigned long long b = 0;
    for (int i = 0; i < NS; ++i) b += 1ULL << (DB * i + DB - 1);
    return b + (1ULL << (DB * NS - 1));  // the top digit has one bit more
}();

template <int PARTS, int LT>
struct TcShape {
    static constexpr int THREADS = LT >= 64 ? 512 : (LT == 32 ? 256 : 128);
    static constexpr int UPT = LT * 16 / THREADS;       // units (line, 8 columns) a thread holds
    // Digits: bytes between 8-column chunks. Core matrices must stay aligned to
    // their 128 bytes (16 bytes of padding here made the products 2x slower).
    static constexpr int LBO = NS * LT * 16;
    static constexpr int PITCH = LT * 8 + 8;            // results: bytes between rows (8 mod 128: banks)
    // accumulator columns of a part (LT = 8: a place more, see consume)
    static constexpr int REGION = LT == 8 ? 8 * LT : kOrders * LT;
    __host__ __device__ static constexpr int part_bytes(int kp) { return kp / 8 * LBO; }
    // Ring of operator blocks: what shared memory the digits leave, at most 24
    // blocks. A block's copy from L2 takes 1300 to 1800 cycles, so narrow tiles,
    // whose products are short, want many in flight.
    static constexpr int RING_OFFSET = PARTS * part_bytes(128);
    static constexpr int STAGES = (231000 - RING_OFFSET) / (int)kBlock < 24 ? (231000 - RING_OFFSET) / (int)kBlock : 24;
    static constexpr int SMEM = RING_OFFSET + STAGES * (int)kBlock;
};

template <int J>
struct Place {
    static constexpr int value = J;
};

// A value of a line whose largest one has the exponent field E, in units of
// 2^(E - 1082): at most 2^60, the grid far below the FP64 rounding of the
// line's largest values.
__device__ __forceinline__ long long tc_fixed(double v, int E) {
    const int hi = __double2hiint(v);
    const int ex = (hi >> 20) & 0x7ff;
    const unsigned mh = (hi & 0xfffff) | (ex ? 0x100000u : 0u);
    const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(v)) << 8;
    int sh = E - (ex ? ex : 1);
    sh = sh > 63 ? 63 : sh;
    const long long f = (long long)(((m >> sh) + 1) >> 1);
    return hi < 0 ? -f : f;
}

// Back to FP64, rounded to nearest (ties away). E >= 64: the result is normal.
__device__ __forceinline__ double tc_to_double(long long y, int E) {
    if (y == 0) return 0.0;
    const unsigned long long m = y < 0 ? 0ULL - (unsigned long long)y : (unsigned long long)y;
    const int lz = __clzll((long long)m);
    const unsigned long long t = (((m << lz) >> 10) + 1) >> 1;  // 2^52 .. 2^53
    const int e = E + 3 - lz;                                   // exponent field less one
    const long long bits = e >= 2046 ? 0x7ff0000000000000LL : (long long)t + ((long long)e << 52);
    return __longlong_as_double(bits | (y & (long long)0x8000000000000000ULL));
}

// The eight biased values F[0..7] of one line and chunk -> six FP16 digits each
// (the lowest at bit SB), stored as 16-byte rows of the B operand (row = place *
// LT + line).
template <int LT, int SB>
__device__ __forceinline__ void tc_put_digits(unsigned char* chunk, int line, const unsigned long long (&F)[8]) {
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        const int sh = SB + DB * (NS - 1 - q);
        const unsigned mask = q == 0 ? 0x7ffu : 0x1ffu;
        const unsigned short off = q == 0 ? 0x6600 : 0x6500;  // 1024 + 512, 1024 + 256
        uint32_t w[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const unsigned a = (unsigned)(F[2 * p] >> sh) & mask;
            const unsigned b = (unsigned)(F[2 * p + 1] >> sh) & mask;
            const unsigned h = (a | (b << 16)) + 0x64006400u;  // 1024 + field, twice
            const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(off)));
            w[p] = *reinterpret_cast<const uint32_t*>(&d);
        }
        const int r = q * LT + line;
        *reinterpret_cast<uint4*>(chunk + (r >> 3) * 128 + (r & 7) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// The order sums of one output -> the 64-bit integer sum in units of 2^-6 of
// order 6.
__device__ __forceinline__ long long tc_combine(const float (&a)[kOrders]) {
    const long long hi = (long long)__float2int_rn(a[0]) * (1 << 18) + (long long)__float2int_rn(a[1]) * (1 << 9) +
                         __float2int_rn(a[2]);
    const int r = __float2int_rn(a[5] * 0.125f);
    const long long lo = (long long)__float2int_rn(a[3]) * (1 << 15) + (long long)__float2int_rn(a[4]) * 64 + r;
    return (hi << 24) + lo;
}

struct TcArgs {
    PassArgs a;
    const unsigned char* img;
    long long lines, ntiles;
    int n, rows, kp, scale, headroom;
    JqFixed jin, jout;
};

template <int PARTS, int LT, bool STRIDED>
__global__ void __launch_bounds__(TcShape<PARTS, LT>::THREADS, 1) tc_pass_kernel(const TcArgs g) {
    using Sh = TcShape<PARTS, LT>;
    constexpr int NT = Sh::THREADS, UPT = Sh::UPT, STAGES = Sh::STAGES, LBO = Sh::LBO;
    constexpr int VPU = PARTS == 2 ? 16 : 8;  // values of a unit
    constexpr bool TWO_PHASES = PARTS == 2 && LT >= 64;
    constexpr int PHASES = TWO_PHASES ? 2 : 1;
    constexpr uint32_t COLS = LT >= 64 ? 512 : (PARTS * Sh::REGION <= 64 ? 64 : PARTS * Sh::REGION <= 128 ? 128
                                               : PARTS * Sh::REGION <= 256 ? 256 : 512);
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_done, bar_never;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ unsigned s_max[LT];

    const PassArgs& a = g.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = g.n, rows = g.rows, kp = g.kp, nkc = kp >> 5;
    const int part_bytes = Sh::part_bytes(kp);
    unsigned char* ring = smem + Sh::RING_OFFSET;
    const double* src = static_cast<const double*>(a.u);
    double* dst = static_cast<double*>(a.u) + a.out_shift;

    if (warp == 0) tmem_alloc(&s_tmem, COLS);
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&bar_full[i], 1);
            mbar_init(&bar_empty[i], 1);
        }
        mbar_init(&bar_done, 1);
        mbar_init(&bar_never, 1);
        s_abort = 0;
        fence_mbar_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = s_tmem;

    // Waits are bounded: a wait that runs out (or another thread's that did)
    // makes the CTA leave its tiles.
    auto wait = [&](uint64_t* bar, unsigned parity) -> bool {
        if (mbar_try_wait(bar, parity)) return true;
        const long long t0 = clock64();
        while (!mbar_try_wait(bar, parity)) {
            if (*reinterpret_cast<volatile int*>(&s_abort)) return false;
            if (clock64() - t0 > a.wait_cycles) {
                *reinterpret_cast<volatile int*>(&s_abort) = 1;
                return false;
            }
        }
        return true;
    };

    // Ring of operator blocks, in the order part, 32-column step, digit place.
    // Blocks are counted modulo the ring only (one thread issues, one thread
    // consumes: a 64-bit division in either loop cost more than the products).
    const int phase_chunks = (TWO_PHASES ? 1 : PARTS) * nkc * NS;
    const int tile_chunks = PARTS * nkc * NS;
    const long long my_tiles = (g.ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
    long long to_produce = my_tiles * tile_chunks;  // thread 32: blocks not issued yet
    int p_stage = 0, p_chunk = 0;                   // thread 32: next stage, block of the tile
    unsigned p_parity = 1;                          // of bar_empty: the first round passes at once
    int c_stage = 0;                                // thread 0: next stage
    unsigned c_parity = 0;
    auto produce = [&](int count) -> bool {
        for (; count > 0 && to_produce > 0; --count, --to_produce) {
            if (!wait(&bar_empty[p_stage], p_parity)) return false;
            mbar_expect_tx(&bar_full[p_stage], kBlock);
            bulk_load(ring + p_stage * kBlock, g.img + (size_t)p_chunk * kBlock, kBlock, &bar_full[p_stage]);
            if (++p_chunk == tile_chunks) p_chunk = 0;
            if (++p_stage == STAGES) {
                p_stage = 0;
                p_parity ^= 1u;
            }
        }
        return true;
    };
    // One 8 KB block: D's digit place J against the places of x, K = 32.
    const uint64_t a_desc0 = tc_desc(smem_u32(ring), 2048, 128), b_desc0 = tc_desc(smem_u32(smem), LBO, 128);
    auto consume = [&](auto place, uint32_t d0, uint64_t bd, bool first) -> bool {
        constexpr int J = decltype(place)::value;
        constexpr int M = 7 - J;  // places of x: orders J + 1 .. 7
        // a first MMA of up to W places, then the rest; N is a multiple of 16, so
        // LT = 8 takes an even number of places, whose last may go to an unused order
        constexpr int W = LT >= 64 ? (M < 4 ? M : 4) : (LT == 8 ? (M + 1) / 2 * 2 : M);
        if (!wait(&bar_full[c_stage], c_parity)) return false;
        const uint64_t ad = a_desc0 + (uint32_t)c_stage * (kBlock >> 4);
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            const uint64_t b0 = bd + ks * (2 * LBO >> 4);
            // place 1 reaches every order: its first products overwrite them
            const uint32_t acc = (J == 1 && ks == 0 && first) ? 0u : 1u;
            tc_mma_f16(d0 + (J - 1) * LT, ad + ks * (4096 >> 4), b0, tc_idesc_f16(128, W * LT), acc);
            if constexpr (M > W)
                tc_mma_f16(d0 + (J - 1 + W) * LT, ad + ks * (4096 >> 4), b0 + (W * LT * 16 >> 4),
                           tc_idesc_f16(128, (M - W) * LT), acc);
        }
        tc_commit(&bar_empty[c_stage]);
        if (++c_stage == STAGES) {
            c_stage = 0;
            c_parity ^= 1u;
        }
        return true;
    };
    if (tid == 32) produce(STAGES);

    unsigned done_parity = 0;
    bool alive = true;
    for (long long tile = blockIdx.x; tile < g.ntiles; tile += gridDim.x) {
        // ---- load: units (line, chunk c of 8 columns, and their mirror images) ----
        for (int i = tid; i < LT; i += NT) s_max[i] = 0;
        __syncthreads();
        double x[UPT][VPU];  // then, as integers, the fixed-point values
        int uline[UPT], uc[UPT];
        const int nch = kp >> 3;
#pragma unroll
        for (int it = 0; it < UPT; ++it) {
            const int u = tid + it * NT;
            // strided axis: lanes along the lines; contiguous axis: a warp takes
            // 4 chunks (256 bytes) of 8 lines
            const int line = STRIDED ? u % LT : (u / 32) % (LT / 8) * 8 + (u & 7);
            const int c = STRIDED ? u / LT : (u / 32) / (LT / 8) * 4 + ((u >> 3) & 3);
            uline[it] = line;
            uc[it] = c;
            const bool in_tile = c < nch;
            if (!in_tile) uline[it] = -1;
            const long long L = tile * LT + line;
#pragma unroll
            for (int r = 0; r < VPU; ++r) x[it][r] = 0.0;
            if (in_tile && L < g.lines) {
                if constexpr (STRIDED) {
                    const long long o = L / a.inner, i = L - o * a.inner;
                    const double* p = src + o * n * a.inner + i;
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const int k = 8 * c + r;
                        if (k < rows) {
                            x[it][r] = p[(long long)k * a.inner];
                            if constexpr (PARTS == 2) x[it][8 + r] = p[(long long)(n - 1 - k) * a.inner];
                        }
                    }
                } else {
                    const double* p = src + L * n;
                    if ((n & 1) == 0 && 8 * c + 8 <= rows) {
#pragma unroll
                        for (int r = 0; r < 8; r += 2) {
                            const double2 v = *reinterpret_cast<const double2*>(p + 8 * c + r);
                            x[it][r] = v.x;
                            x[it][r + 1] = v.y;
                            if constexpr (PARTS == 2) {
                                const double2 w = *reinterpret_cast<const double2*>(p + n - 2 - 8 * c - r);
                                x[it][8 + r] = w.y;
                                x[it][9 + r] = w.x;
                            }
                        }
                    } else {
#pragma unroll
                        for (int r = 0; r < 8; ++r) {
                            const int k = 8 * c + r;
                            if (k < rows) {
                                x[it][r] = p[k];
                                if constexpr (PARTS == 2) x[it][8 + r] = p[n - 1 - k];
                            }
                        }
                    }
                }
            }
            if (a.jq_in) {
#pragma unroll
                for (int r = 0; r < VPU; ++r) x[it][r] = jq_flow_fixed(x[it][r], g.jin);
            }
            unsigned m = 0;
#pragma unroll
            for (int r = 0; r < VPU; ++r) m = max(m, (unsigned)__double2hiint(x[it][r]) & 0x7fffffffu);
            if (in_tile) atomicMax(&s_max[line], m);
        }
        __syncthreads();
        // ---- digits ----
        const int Emin = max(1, 64 - g.scale);
#pragma unroll
        for (int it = 0; it < UPT; ++it) {
            if (uline[it] < 0) continue;
            const int E = max((int)(s_max[uline[it]] >> 20), Emin) + g.headroom;
            unsigned char* chunk = smem + uc[it] * LBO;
#pragma unroll
            for (int r = 0; r < VPU; ++r) x[it][r] = __longlong_as_double(tc_fixed(x[it][r], E));
            // sums and differences in units of 2^(E - 1075), values themselves in
            // units of 2^(E - 1076): at most 2^54 in size, rounded
            constexpr int SB = PARTS == 2 ? 7 : 6;
            constexpr unsigned long long bias = (kBias << SB) + (1ULL << (SB - 1));
            unsigned long long F[8];
            if constexpr (PARTS == 2) {
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    F[r] = bias + __double_as_longlong(x[it][r]) + __double_as_longlong(x[it][8 + r]);
                tc_put_digits<LT, SB>(chunk, uline[it], F);
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    F[r] = bias + __double_as_longlong(x[it][r]) - __double_as_longlong(x[it][8 + r]);
                tc_put_digits<LT, SB>(chunk + part_bytes, uline[it], F);
            } else {
#pragma unroll
                for (int r = 0; r < 8; ++r) F[r] = bias + __double_as_longlong(x[it][r]);
                tc_put_digits<LT, SB>(chunk, uline[it], F);
            }
        }
        fence_proxy_async_smem();
        __syncthreads();

#pragma unroll 1
        for (int ph = 0; ph < PHASES; ++ph) {
            // ---- products ----
            if (tid == 0) {
                tc_fence_after_sync();
                bool ok = true;
                if (a.hold && tile == blockIdx.x && ph == 0) ok = wait(&bar_never, 0);
#pragma unroll 1
                for (int part = TWO_PHASES ? ph : 0; ok && part < (TWO_PHASES ? ph + 1 : PARTS); ++part) {
                    const uint32_t d0 = tmem + (TWO_PHASES ? 0 : part * Sh::REGION);
                    uint64_t bd = b_desc0 + (uint32_t)(part * part_bytes >> 4);
#pragma unroll 1
                    for (int kc = 0; ok && kc < nkc; ++kc, bd += 4 * LBO >> 4)
                        ok = consume(Place<1>(), d0, bd, kc == 0) && consume(Place<2>(), d0, bd, kc == 0) &&
                             consume(Place<3>(), d0, bd, kc == 0) && consume(Place<4>(), d0, bd, kc == 0) &&
                             consume(Place<5>(), d0, bd, kc == 0) && consume(Place<6>(), d0, bd, kc == 0);
                }
                tc_commit(&bar_done);
            } else if (tid == 32) {
                produce(phase_chunks);
            }
            __syncwarp();
            if (!wait(&bar_done, done_parity)) alive = false;
            done_parity ^= 1;
            if (!__syncthreads_and(alive && !*reinterpret_cast<volatile int*>(&s_abort))) {
                alive = false;
                break;
            }
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
                    uint32_t t[kOrders][4];
#pragma unroll
                    for (int s = 0; s < kOrders; ++s) tmem_ld4(taddr + s * LT + cc, t[s]);
                    tc_wait_ld();
                    long long v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float f[kOrders];
#pragma unroll
                        for (int s = 0; s < kOrders; ++s) f[s] = __uint_as_float(t[s][q]);
                        v[q] = tc_combine(f);
                    }
                    long long w[4];
                    if constexpr (PARTS == 2 && !TWO_PHASES) {
#pragma unroll
                        for (int s = 0; s < kOrders; ++s) tmem_ld4(taddr + Sh::REGION + s * LT + cc, t[s]);
                        tc_wait_ld();
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float f[kOrders];
#pragma unroll
                            for (int s = 0; s < kOrders; ++s) f[s] = __uint_as_float(t[s][q]);
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
            __syncthreads();
        }
        if (!alive) break;
        // ---- y = x + D x, the closing flow, store ----
#pragma unroll
        for (int it = 0; it < UPT; ++it) {
            const int line = uline[it], c = uc[it];
            const long long L = tile * LT + line;
            if (line < 0 || L >= g.lines) continue;
            const int Eb = (int)(s_max[line] >> 20);
            const int E = max(Eb, Emin) + g.headroom;
            // the sums are in units of 2^(E - 1082 + f)
            const int left = max(g.scale, 0), right = min(max(-g.scale, 0), 62);
            const long long half = right > 0 ? 1LL << (right - 1) : 0;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int off = (8 * c + r) * Sh::PITCH + line * 8;
                const long long v = *reinterpret_cast<const long long*>(smem + off);
                x[it][r] = tc_to_double(__double_as_longlong(x[it][r]) + ((v << left) + half >> right), E);
                if constexpr (PARTS == 2) {
                    const long long w = *reinterpret_cast<const long long*>(smem + part_bytes + off);
                    x[it][8 + r] = tc_to_double(__double_as_longlong(x[it][8 + r]) + ((w << left) + half >> right), E);
                }
            }
            if (Eb == 2047) {  // a line that holds an infinity or a NaN
#pragma unroll
                for (int r = 0; r < VPU; ++r) x[it][r] = __longlong_as_double(0x7ff8000000000000LL);
            }
            if (a.jq_out) {
#pragma unroll
                for (int r = 0; r < VPU; ++r) x[it][r] = jq_flow_fixed(x[it][r], g.jout);
            }
            if constexpr (STRIDED) {
                const long long o = L / a.inner, i = L - o * a.inner;
                double* p = dst + o * n * a.inner + i;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int k = 8 * c + r;
                    if (k < rows) {
                        p[(long long)k * a.inner] = x[it][r];
                        if constexpr (PARTS == 2) p[(long long)(n - 1 - k) * a.inner] = x[it][8 + r];
                    }
                }
            } else {
                double* p = dst + L * n;
                if ((n & 1) == 0 && 8 * c + 8 <= rows) {
#pragma unroll
                    for (int r = 0; r < 8; r += 2) {
                        *reinterpret_cast<double2*>(p + 8 * c + r) = make_double2(x[it][r], x[it][r + 1]);
                        if constexpr (PARTS == 2)
                            *reinterpret_cast<double2*>(p + n - 2 - 8 * c - r) =
                                make_double2(x[it][9 + r], x[it][8 + r]);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const int k = 8 * c + r;
                        if (k < rows) {
                            p[k] = x[it][r];
                            if constexpr (PARTS == 2) p[n - 1 - k] = x[it][8 + r];
                        }
                    }
                }
            }
        }
        __syncthreads();  // results and s_max are rewritten by the next tile
    }

    if (!alive) {
        // a wait ran out: let this CTA's copies and products in flight finish
        // (bounded), record the timeout
        if (tid == 32) {
            // the copies issued last, one a stage at most: each one's phase of bar_full
            // is the one before the phase its stage would be issued for next
            for (int st = 0; st < STAGES; ++st) {
                const unsigned next = st < p_stage ? p_parity ^ 1u : p_parity;  // bar_empty parity of its next use
                mbar_wait_bounded(&bar_full[st], next, a.wait_cycles);
            }
            if (a.status) atomicOr(a.status, SFAC_PASS_TIMEOUT);
        }
        if (tid == 0) mbar_wait_bounded(&bar_done, done_parity ^ 1u, a.wait_cycles);
        __syncwarp();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, COLS);
}

template <int PARTS, int LT, bool STRIDED>
cudaError_t launch_tc(const TcAxis& ax, const PassArgs& a, long long lines, cudaStream_t s) {
    using Sh = TcShape<PARTS, LT>;
    auto kern = tc_pass_kernel<PARTS, LT, STRIDED>;
    // shared memory is sized for the largest operator, so that one attribute and
    // one resident count hold for every kp (and tensor memory suffices for them)
    const size_t smem_max = Sh::SMEM;
    static LaunchSetup setup;
    int dev = 0, resident = 0;
    cudaError_t err = set_smem(kern, smem_max, setup, &dev);
    if (err == cudaSuccess) err = resident_grid(kern, Sh::THREADS, smem_max, setup, dev, &resident);
    if (err != cudaSuccess) return err;
    TcArgs g;
    g.a = a;
    g.img = static_cast<const unsigned char*>(ax.img);
    g.lines = lines;
    g.ntiles = (lines + LT - 1) / LT;
    g.n = ax.n;
    g.rows = ax.rows;
    g.kp = ax.kp;
    g.scale = ax.scale;
    g.headroom = ax.headroom;
    g.jin = make_jq_fixed(a.jq_in_E, a.jq_in_1mE);
    g.jout = make_jq_fixed(a.jq_out_E, a.jq_out_1mE);
    if (g.ntiles <= 0) return cudaSuccess;
    const long long grid = g.ntiles < resident ? g.ntiles : resident;
    kern<<<(unsigned)grid, Sh::THREADS, smem_max, s>>>(g);
    return cudaGetLastError();
}

template <int PARTS, int LT>
cudaError_t launch_tc_axis(const TcAxis& ax, const PassArgs& a, long long lines, cudaStream_t s) {
    return a.inner > 1 ? launch_tc<PARTS, LT, true>(ax, a, lines, s) : launch_tc<PARTS, LT, false>(ax, a, lines, s);
}

template <int PARTS>
cudaError_t launch_tc_parts(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    const long long lines = a.outer * a.inner;
    const int sms = current_device_sms();
    // the widest tile that still gives every SM one
    if (lines >= 64LL * sms) return launch_tc_axis<PARTS, 64>(ax, a, lines, s);
    if (lines >= 32LL * sms) return launch_tc_axis<PARTS, 32>(ax, a, lines, s);
    if (lines >= 16LL * sms) return launch_tc_axis<PARTS, 16>(ax, a, lines, s);
    return launch_tc_axis<PARTS, 8>(ax, a, lines, s);
}

}  // namespace

cudaError_t launch_pass_tc_f64(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    return ax.parts == 2 ? launch_tc_parts<2>(ax, a, s) : launch_tc_parts<1>(ax, a, s);
}

}  // namespace sfac
