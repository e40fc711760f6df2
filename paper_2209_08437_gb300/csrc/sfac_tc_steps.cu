// sfac_tc_steps.cu - FP64 tensor-core passes with few lines: tiles of 8 lines, and a
// whole sfac_step call on a small grid in one launch.
//
// With at most 8 lines an SM the latency of one tile bounds a pass: load,
// digits, products, sums, store. The arithmetic is that of sfac_tc_tile.cuh; what
// differs is the code: a thread works on pairs of columns in rolled loops and
// the lines' values stay in shared memory, so that the whole pass is a few KB
// of instructions (with the unrolled tile, executed once a pass, instruction
// fetch took more than half of the time: 12,000 cycles for 2D 64^2).
//
// Whole calls: as in sfac_steps.cu a cooperative launch runs every step of the
// call and the CTAs meet at a grid-wide barrier between axis passes. The
// operators do not depend on the field, so the warp that streams them runs
// ahead, through the barriers, by up to 168 KB: the products of a pass find
// their operator in shared memory.
#include <cuda_runtime.h>

#include <atomic>

#include "sfac_tc_tile.cuh"

namespace sfac {
namespace {

constexpr int kLT = 8;
using Shape2 = TcShape<2, kLT>;
constexpr int kNT = 256;  // computing threads; one more warp issues the copies
// Shared memory: digits (then results), the lines' values, the ring.
constexpr int kXArea = Shape2::RING_OFFSET;                  // 2 parts x 64 pairs x 8 lines x 16 bytes
constexpr int kRing = kXArea + 2 * 64 * 128;
constexpr int kG = 3, kStages = 7;  // a stage: kG blocks
constexpr int kSmem = kRing + kStages * kG * (int)kTcBlock;
static_assert(kStages <= kTcMaxStages && kSmem <= 231000, "shared memory");

struct TcStepsArgs {
    TcPass ax[3];
    const unsigned char* img[3];
    int parts[3];
    int dim;
    int single;  // one pass, ax[0], with the flows its own flags ask for; no barrier
    long long nsteps;
    JqFixed half, full;
    unsigned int* bar;
    unsigned int* status;
    long long wait_cycles;
    int hold;
};

// Grid-wide barrier among the computing threads: false if this CTA's wait ran out.
// The counter only grows (reset by the launch): a barrier is passed when it
// reaches `target`, the arrivals of all CTAs so far. One release and one acquire
// are the only round trips to L2.
__device__ __forceinline__ bool tc_grid_barrier(const TcStepsArgs& g, unsigned target, bool held) {
    bool ok = true;
    tc_sync<kNT>();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(g.bar) : "memory");
        if (held) target += 1u << 30;  // the hook: a count that never comes
        const long long t0 = clock64();
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(g.bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if (clock64() - t0 > g.wait_cycles) {
                ok = false;
                break;
            }
        }
    }
    return tc_sync_and<kNT>(ok);
}

// One tile of 8 lines by the computing threads: false if a wait ran out.
template <int PARTS>
__device__ __forceinline__ bool tc_small_tile(const TcPass& g, long long tile, unsigned char* smem, long long* base,
                                              unsigned* smax, TcShared& sh, TcState& st, uint32_t tmem,
                                              long long limit) {
    using Sh = TcShape<PARTS, kLT>;
    constexpr int V = 2 * PARTS, PITCH = Sh::PITCH;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int n = g.n, rows = g.rows, kp = g.kp, units = 4 * kp;  // a unit: a line and a pair of columns
    const int part_bytes = Sh::part_bytes(kp);
    const long long inner = g.inner;
    double2* xs = reinterpret_cast<double2*>(smem + kXArea);

    if (tid < kLT) {
        const long long L = tile * kLT + tid;
        smax[tid] = 0;
        base[tid] = L >= g.lines ? -1 : (inner == 1 ? L * n : L / inner * n * inner + L % inner);
    }
    tc_sync<kNT>();
    // ---- load ----
#pragma unroll 1
    for (int u = tid; u < units; u += kNT) {
        const int line = u & 7, k = u >> 3 << 1;
        const long long b = base[line];
        double v[V];
#pragma unroll
        for (int r = 0; r < V; ++r) v[r] = 0.0;
        if (b >= 0) {
            const double* p = g.src + b;
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (k + r < rows) {
                    v[r] = __ldcg(p + (k + r) * inner);
                    if constexpr (PARTS == 2) v[2 + r] = __ldcg(p + (n - 1 - k - r) * inner);
                }
        }
        if (g.jq_in) jq_flow_fixed_all(v, g.jin);
        unsigned m = 0;
#pragma unroll
        for (int r = 0; r < V; ++r) m = max(m, (unsigned)__double2hiint(v[r]) & 0x7fffffffu);
        xs[u] = make_double2(v[0], v[1]);
        if constexpr (PARTS == 2) xs[512 + u] = make_double2(v[2], v[3]);
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
        if (lane < 8) atomicMax(&smax[line], m);
    }
    tc_sync<kNT>();
    // ---- digits ----
#pragma unroll 1
    for (int u = tid; u < units; u += kNT) {
        const int line = u & 7, k = u >> 3 << 1;
        const int E = tc_scale_of((int)(smax[line] >> 20), g.headroom);
        constexpr int SB = PARTS == 2 ? 7 : 6;
        constexpr unsigned long long bias = (kTcBias << SB) + (1ULL << (SB - 1));
        const double2 v = xs[u];
        const long long a0 = tc_fixed(v.x, E), a1 = tc_fixed(v.y, E);
        xs[u] = make_double2(__longlong_as_double(a0), __longlong_as_double(a1));
        unsigned char* row = smem + (k >> 3) * Sh::LBO + line * 16 + (k & 7) * 2;
        if constexpr (PARTS == 2) {
            const double2 w = xs[512 + u];
            const long long b0 = tc_fixed(w.x, E), b1 = tc_fixed(w.y, E);
            xs[512 + u] = make_double2(__longlong_as_double(b0), __longlong_as_double(b1));
            const unsigned long long s0 = bias + a0 + b0, s1 = bias + a1 + b1;
            const unsigned long long d0 = bias + a0 - b0, d1 = bias + a1 - b1;
#pragma unroll
            for (int q = 0; q < kTcSlices; ++q) {
                *reinterpret_cast<uint32_t*>(row + q * 128) = tc_digit_pair<SB>(s0, s1, q);
                *reinterpret_cast<uint32_t*>(row + part_bytes + q * 128) = tc_digit_pair<SB>(d0, d1, q);
            }
        } else {
#pragma unroll
            for (int q = 0; q < kTcSlices; ++q)
                *reinterpret_cast<uint32_t*>(row + q * 128) = tc_digit_pair<SB>(bias + a0, bias + a1, q);
        }
    }
    fence_proxy_async_smem();
    tc_sync<kNT>();
    // ---- products: the other warps wait at the barrier, not polling ----
    bool ok = true;
    if (warp == 0) {
        tc_fence_after_sync();
        tc_products<PARTS, kLT, kStages, kG>(sh, st, smem, smem + kRing, tmem, 0, PARTS, kp, limit);
        ok = tc_wait(&sh.done, st.done_parity, limit, &sh.abort);
    }
    st.done_parity ^= 1u;
    if (!tc_sync_and<kNT>(ok && *reinterpret_cast<volatile int*>(&sh.abort) == 0)) return false;
    tc_fence_after_sync();
    // ---- the order sums -> integers (row, line): a warp takes 32 rows and 4 lines ----
    {
        const int row = (warp & 3) * 32 + lane, cc = (warp >> 2) * 4;
        const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + cc;
        long long v[PARTS][4];
#pragma unroll
        for (int p = 0; p < PARTS; ++p) {
            uint32_t t[kTcOrders][4];
#pragma unroll
            for (int s = 0; s < kTcOrders; ++s) tmem_ld4(taddr + p * Sh::REGION + s * kLT, t[s]);
            tc_wait_ld();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float f[kTcOrders];
#pragma unroll
                for (int s = 0; s < kTcOrders; ++s) f[s] = __uint_as_float(t[s][q]);
                v[p][q] = tc_combine(f);
            }
        }
        if (row < kp) {
            long long* r0 = reinterpret_cast<long long*>(smem + row * PITCH) + cc;
            long long* r1 = reinterpret_cast<long long*>(smem + part_bytes + row * PITCH) + cc;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if constexpr (PARTS == 2) {
                    r0[q] = v[0][q] + v[1][q];
                    r1[q] = v[0][q] - v[1][q];
                } else {
                    r0[q] = v[0][q];
                }
            }
        }
    }
    tc_fence_before_sync();
    tc_sync<kNT>();
    // ---- y = x + D x, the closing flow, store ----
#pragma unroll 1
    for (int u = tid; u < units; u += kNT) {
        const int line = u & 7, k = u >> 3 << 1;
        const long long b = base[line];
        if (b < 0) continue;
        const int Eb = (int)(smax[line] >> 20);
        const double2 a = xs[u];
        double v[V] = {a.x, a.y};
        if constexpr (PARTS == 2) {
            const double2 w = xs[512 + u];
            v[2] = w.x;
            v[3] = w.y;
        }
        auto cell = [&](int r) {
            return reinterpret_cast<double*>(smem + (r >> 1) * part_bytes + (k + (r & 1)) * PITCH + line * 8);
        };
#pragma unroll
        for (int r = 0; r < V; ++r)
            v[r] = __longlong_as_double(__double_as_longlong(v[r]) + tc_align(__double_as_longlong(*cell(r)), g.scale));
        tc_to_doubles(v, g.headroom, [=](int) { return Eb; }, cell);
        if (g.jq_out) jq_flow_fixed_all(v, g.jout);
        double* p = g.dst + b;
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (k + r < rows) {
                p[(k + r) * inner] = v[r];
                if constexpr (PARTS == 2) p[(n - 1 - k - r) * inner] = v[2 + r];
            }
    }
    return true;
}

__global__ void __launch_bounds__(kNT + 32, 1) tc_steps_kernel(const TcStepsArgs g) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TcShared sh;
    __shared__ unsigned smax[kLT];
    __shared__ long long base[kLT];
    __shared__ TcPass pass;
    if (g.single) pass_next_may_start();
    const uint32_t tmem = tc_setup<Shape2::COLS, kStages>(sh);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    TcState st;
    bool alive = true;
    if (warp == kNT / 32) {
        st.parity = 1;
        long long early = g.single ? kStages : -1;
        for (long long s = 0; alive && s < g.nsteps; ++s)
            for (int ax = 0; alive && ax < g.dim; ++ax) {
                const int stages = g.parts[ax] * (g.ax[ax].kp >> 5) * kTcSlices / kG;
                for (long long tile = blockIdx.x; alive && tile < g.ax[ax].ntiles; tile += gridDim.x) {
                    st.left = stages;
                    alive = tc_produce<kStages, kG>(sh, st, smem + kRing, g.img[ax], stages, stages, g.wait_cycles,
                                                    early);
                    early -= stages;
                }
            }
    } else {
        if (g.single) pass_wait_for_previous();
        if (g.single && g.hold && warp == 0) tc_wait(&sh.never, 0, g.wait_cycles, &sh.abort);  // the test hook
        unsigned target = 0;
        for (long long s = 0; alive && s < g.nsteps; ++s) {
            const bool last = s == g.nsteps - 1;
            for (int ax = 0; alive && ax < g.dim; ++ax) {
                // J^Q_{tau/2} opens the first step and closes the last one; between
                // two steps the closing and opening halves act as one J^Q_tau
                if (threadIdx.x == 0) {
                    pass = g.ax[ax];
                    if (!g.single) {
                        pass.jq_in = ax == 0 && s == 0;
                        pass.jin = g.half;
                        pass.jq_out = ax == g.dim - 1;
                        pass.jout = last ? g.half : g.full;
                    }
                }
                tc_sync<kNT>();
                for (long long tile = blockIdx.x; alive && tile < pass.ntiles; tile += gridDim.x) {
                    alive = g.parts[ax] == 2
                                ? tc_small_tile<2>(pass, tile, smem, base, smax, sh, st, tmem, g.wait_cycles)
                                : tc_small_tile<1>(pass, tile, smem, base, smax, sh, st, tmem, g.wait_cycles);
                    if (alive) tc_sync<kNT>();  // base, smax and the results are rewritten by the next tile
                }
                if (alive && !(last && ax == g.dim - 1))
                    alive = tc_grid_barrier(g, target += gridDim.x, g.hold != 0 && s == 0 && ax == 0);
            }
        }
        if (!alive) *reinterpret_cast<volatile int*>(&sh.abort) = 1;  // also ends the producer's waits
    }
    __syncthreads();
    if (sh.abort) {
        if (warp == kNT / 32) tc_drain_copies<kStages>(sh, st, g.wait_cycles);
        if (threadIdx.x == 0) {
            mbar_wait_bounded(&sh.done, st.done_parity ^ 1u, g.wait_cycles);
            if (g.status) atomicOr(g.status, SFAC_PASS_TIMEOUT);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, Shape2::COLS);
}

}  // namespace

namespace {

cudaError_t launch_small(TcStepsArgs& g, const TcAxis* ax, const PassArgs* pa, bool cooperative, cudaStream_t s) {
    static LaunchSetup setup;
    int dev = 0, resident = 0;
    cudaError_t err = set_smem(tc_steps_kernel, kSmem, setup, &dev);
    if (err == cudaSuccess) err = resident_grid(tc_steps_kernel, kNT + 32, kSmem, setup, dev, &resident);
    if (err != cudaSuccess) return err;
    long long grid = 1;
    for (int l = 0; l < g.dim; ++l) {
        g.ax[l] = tc_pass_of<double>(ax[l], pa[l]);
        g.ax[l].ntiles = (g.ax[l].lines + kLT - 1) / kLT;
        g.img[l] = static_cast<const unsigned char*>(ax[l].img);
        g.parts[l] = ax[l].parts;
        grid = g.ax[l].ntiles > grid ? g.ax[l].ntiles : grid;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(grid < resident ? grid : resident));
    cfg.blockDim = dim3(kNT + 32);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (cooperative) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0] = pass_overlap_attribute();
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tc_steps_kernel, g);
}

}  // namespace

cudaError_t launch_tc_steps(const TcAxis* ax, const StepsArgs& a, cudaStream_t s) {
    cudaError_t err = cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned int), s);
    if (err != cudaSuccess) return err;
    TcStepsArgs g;
    g.dim = a.dim;
    g.single = 0;
    g.nsteps = a.nsteps;
    g.half = make_jq_fixed(a.jq_half_E, a.jq_half_1mE);
    g.full = make_jq_fixed(a.jq_full_E, a.jq_full_1mE);
    g.bar = a.bar;
    g.status = a.status;
    g.wait_cycles = a.wait_cycles;
    g.hold = a.hold;
    return launch_small(g, ax, a.ax, true, s);
}

cudaError_t launch_pass_tc_small(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    TcStepsArgs g{};
    g.dim = 1;
    g.single = 1;
    g.nsteps = 1;
    g.status = a.status;
    g.wait_cycles = a.wait_cycles;
    g.hold = a.hold;
    if (a.outer * a.inner <= 0) return cudaSuccess;
    return launch_small(g, &ax, &a, false, s);
}

}  // namespace sfac
