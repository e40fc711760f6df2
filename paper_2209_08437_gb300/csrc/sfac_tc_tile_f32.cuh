// sfac_tc_tile_f32.cuh - FP32 lines as digit products on the tensor cores.
//
// As sfac_tc_tile.cuh, in FP32 precision: three digits of 10 bits of x (30 bits
// of the line's scale) times three of D, orders 2..4 (six products). y = x + D x
// keeps x in FP32, so only the increment sees the fixed point; the order sums are
// combined by FP32 multiply-adds, and the nonlinear flow is the increment form
// of the FP32 passes: y = x0 + (all increments), rounded once.
#pragma once

#include "sfac_tc_tile.cuh"

namespace sfac {

constexpr unsigned kTcBias32 = (1u << 29) + (1u << 19) + (1u << 9);

// Two biased values -> digit place q as two FP16 integers.
__device__ __forceinline__ uint32_t tc_digit_pair32(unsigned f0, unsigned f1, int q) {
    const int sh = kTcBits32 * (kTcSlices32 - 1 - q);
    const unsigned mask = q == 0 ? 0x7ffu : 0x3ffu;
    const unsigned h = (((f0 >> sh) & mask) | (((f1 >> sh) & mask) << 16)) + 0x64006400u;  // 1024 + field
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6600)));
    return *reinterpret_cast<const uint32_t*>(&d);
}

template <int LT>
__device__ __forceinline__ void tc_put_digits32(unsigned char* chunk, int line, const unsigned (&F)[8]) {
#pragma unroll
    for (int q = 0; q < kTcSlices32; ++q) {
        const int r = q * LT + line;
        *reinterpret_cast<uint4*>(chunk + (r >> 3) * 128 + (r & 7) * 16) =
            make_uint4(tc_digit_pair32(F[0], F[1], q), tc_digit_pair32(F[2], F[3], q),
                       tc_digit_pair32(F[4], F[5], q), tc_digit_pair32(F[6], F[7], q));
    }
}

// Eight consecutive values at any 4-byte aligned p, as tc_load8.
__device__ __forceinline__ void tc_load8(const float* p, bool inside, float (&v)[8]) {
    if ((reinterpret_cast<uintptr_t>(p) & 31) == 0) {  // a sector
        asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                     : "l"(p)
                     : "memory");
        return;
    }
    const unsigned s = (unsigned)(reinterpret_cast<uintptr_t>(p) >> 2) & 3u;
    if (s != 0 && !inside) {
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = p[r];
        return;
    }
    const float4* q = reinterpret_cast<const float4*>(p - s);
    float t[12], h[11];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < 2 || s != 0) w = q[i];
        t[4 * i] = w.x, t[4 * i + 1] = w.y, t[4 * i + 2] = w.z, t[4 * i + 3] = w.w;
    }
#pragma unroll
    for (int r = 0; r < 11; ++r) h[r] = s & 1u ? t[r + 1] : t[r];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = s & 2u ? h[r + 2] : h[r];
}
__device__ __forceinline__ void tc_store8(float* p, const float (&v)[8]) {
    if ((reinterpret_cast<uintptr_t>(p) & 31) == 0) {
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                     "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                     : "memory");
        return;
    }
    auto two = [&](int i) { *reinterpret_cast<float2*>(p + i) = make_float2(v[i], v[i + 1]); };
    auto four = [&](int i) { *reinterpret_cast<float4*>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]); };
    switch ((unsigned)(reinterpret_cast<uintptr_t>(p) >> 2) & 3u) {
        case 0: four(0), four(4); break;
        case 1: p[0] = v[0], two(1), four(3), p[7] = v[7]; break;
        case 2: two(0), four(2), two(6); break;
        default: p[0] = v[0], four(1), two(5), p[7] = v[7]; break;
    }
}

// One tile of LT lines, by the computing threads: false if a wait ran out.
template <int PARTS, int LT, bool STRIDED, int STAGES>
__device__ __forceinline__ bool tc_tile_f32(const TcPassT<float>& g, long long tile, unsigned char* smem,
                                            unsigned char* ring, unsigned* smax, TcShared& sh, TcState& st,
                                            uint32_t tmem, const unsigned char* img, int tid, long long limit) {
    using Sh = TcShape<PARTS, LT, kTcSlices32>;
    constexpr int NT = Sh::THREADS, UPT = Sh::UPT, LBO = Sh::LBO;
    constexpr int VPU = PARTS == 2 ? 16 : 8;
    static_assert(!Sh::TWO_PHASES, "both parts' accumulators fit");
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n = g.n, rows = g.rows, kp = g.kp;
    const int part_bytes = Sh::part_bytes(kp);

    // ---- load: units (line, chunk c of 8 columns, and their mirror images) ----
    for (int i = tid; i < LT; i += NT) smax[i] = 0;
    tc_sync<NT>();
    float x[UPT][VPU], d[UPT][VPU];  // x0 and its increments so far
    int uline[UPT], uc[UPT];
    const int nch = kp >> 3;
#pragma unroll
    for (int it = 0; it < UPT; ++it) {
        const int u = tid + it * NT;
        // strided axis: lanes along the lines; contiguous axis: a warp takes
        // 4 chunks (128 bytes) of 8 lines
        const int line = STRIDED ? u % LT : (u / 32) % (LT / 8) * 8 + (u & 7);
        const int c = STRIDED ? u / LT : (u / 32) / (LT / 8) * 4 + ((u >> 3) & 3);
        const bool in_tile = c < nch;
        uline[it] = in_tile ? line : -1;
        uc[it] = c;
        const long long L = tile * LT + line;
#pragma unroll
        for (int r = 0; r < VPU; ++r) x[it][r] = d[it][r] = 0.f;
        if (in_tile && L < g.lines) {
            const long long o = STRIDED ? L / g.inner : L, i = STRIDED ? L - o * g.inner : 0;
            const float* p = g.src + (STRIDED ? o * n * g.inner + i : L * n);
            const long long stride = STRIDED ? g.inner : 1;
            if (!STRIDED && 8 * c + 8 <= rows) {
                float v[8];
                tc_load8(p + 8 * c, tc_groups_inside(L * n + 8 * c, g.lines * n), v);
#pragma unroll
                for (int r = 0; r < 8; ++r) x[it][r] = v[r];
                if constexpr (PARTS == 2) {
                    tc_load8(p + n - 8 - 8 * c, tc_groups_inside(L * n + n - 8 - 8 * c, g.lines * n), v);
#pragma unroll
                    for (int r = 0; r < 8; ++r) x[it][8 + r] = v[7 - r];
                }
            } else {
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int k = 8 * c + r;
                    if (k < rows) {
                        x[it][r] = p[k * stride];
                        if constexpr (PARTS == 2) x[it][8 + r] = p[(n - 1 - k) * stride];
                    }
                }
            }
        }
        if (g.jq_in) {
            const float om = (float)g.jin.omE;
#pragma unroll
            for (int r = 0; r < VPU; ++r) d[it][r] = jq_increment(x[it][r], om);
        }
        unsigned m = 0;
#pragma unroll
        for (int r = 0; r < VPU; ++r) m = max(m, __float_as_uint(x[it][r] + d[it][r]) & 0x7fffffffu);
        if (in_tile) atomicMax(&smax[line], m);
    }
    tc_sync<NT>();
    // ---- digits: x in units of 2^(E - 154) (parts) or 2^(E - 155), sums below 2^29 ----
    // Below E = 28 the factor has no exponent left: a second one, for every line, which
    // costs less than a branch (3D 200^3 x 2: 287 us without, 289, with a branch 293).
    constexpr int Emin = 28;
#pragma unroll
    for (int it = 0; it < UPT; ++it) {
        if (uline[it] < 0) continue;
        const int E = max((int)(smax[uline[it]] >> 23), 1);
        const float m = __uint_as_float((unsigned)((PARTS == 2 ? 281 : 282) - max(E, Emin)) << 23);
        const float up = __uint_as_float((unsigned)(127 + max(Emin - E, 0)) << 23);
        unsigned char* chunk = smem + uc[it] * LBO;
        int X[VPU];
#pragma unroll
        for (int r = 0; r < VPU; ++r) X[r] = __float2int_rn(fmaf(x[it][r], m, d[it][r] * m) * up);
        unsigned F[8];
        if constexpr (PARTS == 2) {
#pragma unroll
            for (int r = 0; r < 8; ++r) F[r] = kTcBias32 + (unsigned)(X[r] + X[8 + r]);
            tc_put_digits32<LT>(chunk, uline[it], F);
#pragma unroll
            for (int r = 0; r < 8; ++r) F[r] = kTcBias32 + (unsigned)(X[r] - X[8 + r]);
            tc_put_digits32<LT>(chunk + part_bytes, uline[it], F);
        } else {
#pragma unroll
            for (int r = 0; r < 8; ++r) F[r] = kTcBias32 + (unsigned)X[r];
            tc_put_digits32<LT>(chunk, uline[it], F);
        }
    }
    fence_proxy_async_smem();
    tc_sync<NT>();
    // ---- products: the other warps wait at the barrier, not polling ----
    bool ok = true;
    if (warp == 0) {
        tc_fence_after_sync();
        tc_products<PARTS, LT, STAGES, Sh::G, kTcSlices32>(sh, st, smem, ring, tmem, 0, PARTS, kp, limit);
        ok = tc_wait(&sh.done, st.done_parity, limit, &sh.abort);
    }
    if (warp >= 2) tc_prefetch<LT, STRIDED>(g, tile + gridDim.x, tid - 64, NT - 64);
    if (!Sh::OWN_PRODUCER && warp == 1)
        tc_produce<STAGES, Sh::G>(sh, st, ring, img, PARTS * (kp >> 5) * kTcSlices32 / Sh::G,
                                  PARTS * (kp >> 5) * kTcSlices32 / Sh::G, limit);
    st.done_parity ^= 1u;
    if (!tc_sync_and<NT>(ok && *reinterpret_cast<volatile int*>(&sh.abort) == 0)) return false;
    tc_fence_after_sync();
    // ---- the order sums, combined, through shared memory (row, line) ----
    {
        constexpr int GROUPS = NT / 128, CPG = LT / GROUPS;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const int col0 = (warp >> 2) * CPG;
        // 2^f, the operator's scale
        const float w2 = __uint_as_float((unsigned)(127 + g.scale) << 23), w3 = w2 * 0x1p-10f, w4 = w2 * 0x1p-20f;
        float* r0 = reinterpret_cast<float*>(smem + row * Sh::PITCH);
        float* r1 = reinterpret_cast<float*>(smem + part_bytes + row * Sh::PITCH);
#pragma unroll 1
        for (int cc = col0; cc < col0 + CPG; cc += 4) {
            __syncwarp();
            uint32_t t[PARTS][kTcSlices32][4];
#pragma unroll
            for (int p = 0; p < PARTS; ++p)
#pragma unroll
                for (int s = 0; s < kTcSlices32; ++s) tmem_ld4(taddr + p * Sh::REGION + s * LT + cc, t[p][s]);
            tc_wait_ld();
            if (row < kp) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float v[PARTS];
#pragma unroll
                    for (int p = 0; p < PARTS; ++p)
                        v[p] = fmaf(__uint_as_float(t[p][2][q]), w4,
                                    fmaf(__uint_as_float(t[p][1][q]), w3, __uint_as_float(t[p][0][q]) * w2));
                    if constexpr (PARTS == 2) {
                        r0[cc + q] = v[0] + v[1];
                        r1[cc + q] = v[0] - v[1];
                    } else {
                        r0[cc + q] = v[0];
                    }
                }
            }
        }
    }
    tc_fence_before_sync();
    tc_sync<NT>();
    // ---- y = x0 + increments, the closing flow, store ----
#pragma unroll
    for (int it = 0; it < UPT; ++it) {
        const int line = uline[it], c = uc[it];
        const long long L = tile * LT + line;
        if (line < 0 || L >= g.lines) continue;
        const int Eb = (int)(smax[line] >> 23);
        // the sums are in units of 2^(E - 145), a subnormal for E < 19; NaN for a line
        // that holds an infinity or a NaN
        const int E = max(Eb, 1);
        const float sc = __uint_as_float(Eb == 255 ? 0x7fc00000u : E > 18 ? (unsigned)(E - 18) << 23 : 16u << E);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int off = (8 * c + r) * Sh::PITCH + line * 4;
            d[it][r] = fmaf(*reinterpret_cast<const float*>(smem + off), sc, d[it][r]);
            if constexpr (PARTS == 2)
                d[it][8 + r] = fmaf(*reinterpret_cast<const float*>(smem + part_bytes + off), sc, d[it][8 + r]);
        }
        if (g.jq_out) {
            const float om = (float)g.jout.omE;
#pragma unroll
            for (int r = 0; r < VPU; ++r) d[it][r] += jq_increment(x[it][r] + d[it][r], om);
        }
#pragma unroll
        for (int r = 0; r < VPU; ++r) x[it][r] += d[it][r];
        const long long o = STRIDED ? L / g.inner : L, i = STRIDED ? L - o * g.inner : 0;
        float* p = g.dst + (STRIDED ? o * n * g.inner + i : L * n);
        const long long stride = STRIDED ? g.inner : 1;
        if (!STRIDED && 8 * c + 8 <= rows) {
            float v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = x[it][r];
            tc_store8(p + 8 * c, v);
            if constexpr (PARTS == 2) {
#pragma unroll
                for (int r = 0; r < 8; ++r) v[r] = x[it][15 - r];
                tc_store8(p + n - 8 - 8 * c, v);
            }
        } else {
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
    tc_sync<NT>();  // results and smax are rewritten by the next tile
    return true;
}

}  // namespace sfac
