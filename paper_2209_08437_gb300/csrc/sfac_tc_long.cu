// sfac_tc_long.cu - FP64 passes of 257 to 1024 points on the tensor cores.
//
// The arithmetic is that of sfac_tc_tile.cuh. A line's digits no longer fit in
// shared memory beside a ring for the operator (n = 1024: 12 KB a line), and one
// CTA would stream the whole operator (6.3 MB) for few lines. Here a cluster
// takes a tile of 32 lines, and each of its CTAs 128 output rows of both halves
// (and their mirror images): a CTA streams only its rows of the operator, while
// every CTA of the cluster converts the whole lines to digits itself, 32 columns
// at a time (converting them again is cheaper than moving the digits: n = 1024,
// about 1,300 cycles a step against 3,600 for streaming the step's operator).
// After every 128 columns the order sums leave tensor memory for 64-bit
// registers, so that they stay exact. The field is updated in place: a cluster
// barrier separates the last load of the lines from the first store.
//
// Eight warps convert, drain and store; one more issues the copies and one the
// products. Measured on 2D 1024^2 (side by side, passes without the flow): 205 us a
// pass by FFTs on the FP64 pipe (90% busy), 62 us contiguous and 54 us strided here;
// 512^2 37 and 33 us. By the times of its parts the loads' latency and the conversion
// bound it.
#include <cuda_runtime.h>

#include <atomic>

#include "sfac_tc_tile.cuh"

namespace sfac {
namespace {

constexpr int kLT = 32;
using Shape = TcShape<2, kLT>;
constexpr int kNT = 256;             // converting threads
constexpr int kThreads = kNT + 64;
constexpr int kStepBytes = Shape::part_bytes(32);  // digits of 32 columns of one part
constexpr int kBuffers = 2;
constexpr int kRing = kBuffers * 2 * kStepBytes;
constexpr int kG = 3, kStages = 7;    // a stage: kG blocks of the operator
constexpr int kSmem = kRing + kStages * kG * (int)kTcBlock;
constexpr int kPitch = kLT * 8 + 8;  // results, in the ring's place: bytes between rows
static_assert(kSmem <= 231000 && kStages <= kTcMaxStages && 2 * 128 * kPitch <= kStages * kG * (int)kTcBlock, "smem");

struct TcLongArgs {
    TcPass pass;
    const unsigned char* img;
    unsigned int* status;
    long long wait_cycles;
    int hold;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// All threads of all CTAs of the cluster.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <bool STRIDED>
__global__ void __launch_bounds__(kThreads, 1) tc_long_kernel(const TcLongArgs g) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TcShared sh;
    __shared__ uint64_t dfull[kBuffers], dfree[kBuffers], drained;
    __shared__ unsigned smax[kLT];
    __shared__ long long sbase[kLT];
    const TcPass& ps = g.pass;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    pass_next_may_start();
    unsigned rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const long long tile = blockIdx.x / ((ps.rows + 127) / 128);
    const int n = ps.n, rows = ps.rows, nkc = ps.kp >> 5;
    const long long limit = g.wait_cycles, inner = ps.inner;
    if (tid < kLT) {
        const long long L = tile * kLT + tid;
        smax[tid] = L >= ps.lines ? 1023u << 20 : 0;  // a missing line is not a rare one (tc_plain)
        sbase[tid] = L >= ps.lines ? -1 : STRIDED ? L / inner * n * inner + L % inner : L * n;
    }
    if (tid == 0) {
        for (int b = 0; b < kBuffers; ++b) {
            mbar_init(&dfull[b], kNT / 32);
            mbar_init(&dfree[b], 1);
        }
        mbar_init(&drained, kNT / 32);
        fence_mbar_init();
    }
    const uint32_t tmem = tc_setup<Shape::COLS, kStages>(sh);

    TcState st;
    bool alive = true;
    if (warp == kNT / 32) {
        // ---- the copies ----
        st.parity = 1;
        st.left = nkc * 2 * kTcSlices / kG;
        const unsigned char* img = g.img + (size_t)rank * nkc * 2 * kTcSlices * kTcBlock;
        tc_produce<kStages, kG>(sh, st, smem + kRing, img, nkc * 2 * kTcSlices / kG, st.left, limit,
                                kStages);
    } else if (warp == kNT / 32 + 1) {
        // ---- the products ----
        pass_wait_for_previous();  // no limit runs before the lines can be loaded (tc_produce)
        if (g.hold) alive = tc_wait(&sh.never, 0, limit, &sh.abort);  // the test hook
        const uint64_t a0 = tc_desc(smem_u32(smem + kRing), 2048, 128), b0 = tc_desc(smem_u32(smem), Shape::LBO, 128);
#pragma unroll 1
        for (int kc = 0; alive && kc < nkc; ++kc) {
            const int buf = kc & 1;
            if ((kc & 3) == 0 && kc > 0)  // the sums of the last 128 columns have been read
                alive = tc_wait(&drained, (unsigned)((kc >> 2) - 1) & 1u, limit, &sh.abort);
            alive = alive && tc_wait(&dfull[buf], (unsigned)(kc >> 1) & 1u, limit, &sh.abort);
            tc_fence_after_sync();
            uint64_t bd = b0 + (uint32_t)(buf * 2 * kStepBytes >> 4);
            int j = 0;
            uint32_t d0 = tmem;
#pragma unroll 1
            for (int b = 0; alive && b < 2 * kTcSlices / kG; ++b) {
                alive = tc_wait(&sh.full[st.stage], st.parity, limit, &sh.abort);
                if (!alive) break;
                uint64_t ad = a0 + (uint32_t)(st.stage * (kG * kTcBlock >> 4));
#pragma unroll 1
                for (int q = 0; q < kG; ++q, ad += kTcBlock >> 4) {
                    const uint32_t idesc = tc_idesc_f16(128, 0) + ((uint32_t)((kTcSlices - j) * kLT) >> 3 << 17);
                    const uint32_t acc = j == 0 && (kc & 3) == 0 ? 0u : 1u;
                    if (elect_one()) {
                        tc_mma_f16(d0 + j * kLT, ad, bd, idesc, acc);
                        tc_mma_f16(d0 + j * kLT, ad + (4096 >> 4), bd + (2 * Shape::LBO >> 4), idesc, 1u);
                        if (q == kG - 1) tc_commit(&sh.empty[st.stage]);
                    }
                    __syncwarp();
                    if (++j == kTcSlices) {
                        j = 0;
                        d0 += Shape::REGION;
                        bd += kStepBytes >> 4;
                    }
                }
                if (++st.stage == kStages) {
                    st.stage = 0;
                    st.parity ^= 1u;
                }
            }
            if (elect_one()) {
                tc_commit(&dfree[buf]);
                if ((kc & 3) == 3 || kc == nkc - 1) tc_commit(&sh.done);
            }
            __syncwarp();
        }
    }
    // ---- converting warps ----
    // strided axis: lanes along the lines; contiguous axis: a warp takes 16
    // columns (128 bytes) of 8 lines. A unit: 4 columns and their mirror images.
    const int line = STRIDED ? lane : (warp & 3) * 8 + (lane & 7);
    const int cg = STRIDED ? warp : (warp >> 2) * 4 + (lane >> 3);
    long long sum[2][16];  // row (warp & 3) * 32 + lane, lines (warp >> 2) * 16 ..
    if (warp < kNT / 32) {
        pass_wait_for_previous();
        const long long base = sbase[line];
        const double* p = ps.src + (base < 0 ? 0 : base);
        auto load = [&](int kc, double (&v)[8]) {
            const int k0 = kc * 32 + cg * 4;
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = 0.0;
            if (base < 0) return;
            if (!STRIDED && (n & 1) == 0 && k0 + 4 <= rows) {
#pragma unroll
                for (int r = 0; r < 4; r += 2) {
                    const double2 a = *reinterpret_cast<const double2*>(p + k0 + r);
                    const double2 b = *reinterpret_cast<const double2*>(p + n - 2 - k0 - r);
                    v[r] = a.x, v[r + 1] = a.y, v[4 + r] = b.y, v[5 + r] = b.x;
                }
                return;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (k0 + r < rows) {
                    v[r] = p[(k0 + r) * inner];
                    v[4 + r] = p[(n - 1 - k0 - r) * inner];
                }
        };
        // the line's largest value
        unsigned m = 0;
#pragma unroll 4
        for (int kc = 0; kc < nkc; ++kc) {
            double v[8];
            load(kc, v);
#pragma unroll
            for (int r = 0; r < 8; ++r) m = max(m, (unsigned)__double2hiint(v[r]) & 0x7fffffffu);
        }
        atomicMax(&smax[line], m);
        tc_sync<kNT>();
        const int E = tc_scale_of((int)(smax[line] >> 20), ps.headroom);
#pragma unroll
        for (int q = 0; q < 16; ++q) sum[0][q] = sum[1][q] = 0;
        double v[8];
        load(0, v);
#pragma unroll 1
        for (int kc = 0; alive && kc < nkc; ++kc) {
            const int buf = kc & 1;
            double cur[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) cur[r] = v[r];
            if (kc + 1 < nkc) load(kc + 1, v);  // the next step's values, while this one is converted
            long long X[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) X[r] = tc_fixed(cur[r], E);
            if (kc >= kBuffers) alive = tc_wait(&dfree[buf], (unsigned)((kc >> 1) - 1) & 1u, limit, &sh.abort);
            constexpr int SB = 7;
            constexpr unsigned long long bias = (kTcBias << SB) + (1ULL << (SB - 1));
            unsigned char* row = smem + buf * 2 * kStepBytes + (cg >> 1) * Shape::LBO + (cg & 1) * 8;
#pragma unroll
            for (int q = 0; q < kTcSlices; ++q) {
                const int rr = q * kLT + line;
                unsigned char* at = row + (rr >> 3) * 128 + (rr & 7) * 16;
                *reinterpret_cast<uint2*>(at) =
                    make_uint2(tc_digit_pair<SB>(bias + X[0] + X[4], bias + X[1] + X[5], q),
                               tc_digit_pair<SB>(bias + X[2] + X[6], bias + X[3] + X[7], q));
                *reinterpret_cast<uint2*>(at + kStepBytes) =
                    make_uint2(tc_digit_pair<SB>(bias + X[0] - X[4], bias + X[1] - X[5], q),
                               tc_digit_pair<SB>(bias + X[2] - X[6], bias + X[3] - X[7], q));
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dfull[buf]);
            if ((kc & 3) == 3 || kc == nkc - 1) {
                // ---- the order sums of these 128 columns -> integers ----
                alive = alive && tc_wait(&sh.done, (unsigned)(kc >> 2) & 1u, limit, &sh.abort);
                if (!alive) break;
                tc_fence_after_sync();
                const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 16;
#pragma unroll
                for (int part = 0; part < 2; ++part)
#pragma unroll
                    for (int cc = 0; cc < 16; cc += 4) {
                        uint32_t t[kTcOrders][4];
#pragma unroll
                        for (int s = 0; s < kTcOrders; ++s) tmem_ld4(taddr + part * Shape::REGION + s * kLT + cc, t[s]);
                        tc_wait_ld();
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float f[kTcOrders];
#pragma unroll
                            for (int s = 0; s < kTcOrders; ++s) f[s] = __uint_as_float(t[s][q]);
                            sum[part][cc + q] += tc_combine(f);
                        }
                    }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&drained);
            }
        }
    }
    // every CTA of the cluster has loaded the lines
    __syncwarp();
    cluster_sync();
    const bool failed = *reinterpret_cast<volatile int*>(&sh.abort) != 0;
    if (warp < kNT / 32 && !failed) {
        // ---- y = x + D x: the sums through shared memory (row, line), in the ring's place ----
        const int row = (warp & 3) * 32 + lane, l0 = (warp >> 2) * 16;
        long long* r0 = reinterpret_cast<long long*>(smem + kRing + row * kPitch) + l0;
        long long* r1 = reinterpret_cast<long long*>(smem + kRing + (128 + row) * kPitch) + l0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            r0[q] = sum[0][q] + sum[1][q];
            r1[q] = sum[0][q] - sum[1][q];
        }
        tc_sync<kNT>();
        // four values and their mirror images at a time, so that their loads overlap
        constexpr int B = 4;
#pragma unroll 1
        for (int u0 = tid; u0 < 128 * kLT; u0 += B * kNT) {
            double v[2 * B];
            auto where = [&](int i, int* rr, int* l) {
                const int u = u0 + i * kNT;
                *rr = STRIDED ? u / kLT : u % 128;
                *l = STRIDED ? u % kLT : u / 128;
                return (int)rank * 128 + *rr < rows ? sbase[*l] : -1;
            };
            auto cell = [&](int i) {  // value i: B values, then their mirror images
                int rr, l;
                where(i % B, &rr, &l);
                return reinterpret_cast<double*>(smem + kRing + (i / B * 128 + rr) * kPitch + l * 8);
            };
#pragma unroll
            for (int i = 0; i < B; ++i) {
                int rr, l;
                const long long b = where(i, &rr, &l);
                const int k = (int)rank * 128 + rr;
                v[i] = b < 0 ? 0.0 : ps.src[b + k * inner];
                v[B + i] = b < 0 ? 0.0 : ps.src[b + (n - 1 - k) * inner];
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                int rr, l;
                where(i, &rr, &l);
                const int E = tc_scale_of((int)(smax[l] >> 20), ps.headroom);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    double& w = v[h * B + i];
                    const long long d = __double_as_longlong(*cell(h * B + i));
                    w = __longlong_as_double(tc_fixed(w, E) + tc_align(d, ps.scale));
                }
            }
            auto field = [&](int r) {
                int rr, l;
                where(r % B, &rr, &l);
                return (int)(smax[l] >> 20);
            };
            tc_to_doubles(v, ps.headroom, field, cell);
            if (ps.jq_out) jq_flow_fixed_all(v, ps.jout);
#pragma unroll
            for (int i = 0; i < B; ++i) {
                int rr, l;
                const long long b = where(i, &rr, &l);
                const int k = (int)rank * 128 + rr;
                if (b < 0) continue;
                ps.dst[b + k * inner] = v[i];
                ps.dst[b + (n - 1 - k) * inner] = v[B + i];
            }
        }
    }
    __syncthreads();
    if (sh.abort) {
        // a wait ran out: let the copies and products in flight finish, record it
        if (warp == kNT / 32) tc_drain_copies<kStages>(sh, st, limit);
        if (warp == kNT / 32 + 1) {
            if (elect_one()) tc_commit(&sh.never);
            __syncwarp();
            if (lane == 0) mbar_wait_bounded(&sh.never, 0, limit);
        }
        if (tid == 0 && g.status) atomicOr(g.status, SFAC_PASS_TIMEOUT);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, Shape::COLS);
}

// The opening flow, value by value, as a launch of its own: inside the pass every
// CTA of the cluster and the closing update would each apply it again (2D
// 1024^2: 96 us a pass, against 62 us without the flow).
__global__ void __launch_bounds__(256) tc_flow_kernel(const double* src, double* dst, long long npts, JqFixed q) {
    pass_next_may_start();
    pass_wait_for_previous();
    constexpr int V = 4;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < npts; i += V * stride) {
        double v[V];
#pragma unroll
        for (int r = 0; r < V; ++r) v[r] = i + r * stride < npts ? src[i + r * stride] : 0.0;
        jq_flow_fixed_all(v, q);
#pragma unroll
        for (int r = 0; r < V; ++r)
            if (i + r * stride < npts) dst[i + r * stride] = v[r];
    }
}

template <bool STRIDED>
cudaError_t launch_long(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    static LaunchSetup setup;
    int dev = 0;
    cudaError_t err = set_smem(tc_long_kernel<STRIDED>, kSmem, setup, &dev);
    if (err != cudaSuccess) return err;
    TcLongArgs g;
    g.pass = tc_pass_of<double>(ax, a);
    g.pass.ntiles = (g.pass.lines + kLT - 1) / kLT;
    g.img = static_cast<const unsigned char*>(ax.img);
    g.status = a.status;
    g.wait_cycles = a.wait_cycles;
    g.hold = a.hold;
    const int cluster = (ax.rows + 127) / 128;
    if (g.pass.ntiles <= 0) return cudaSuccess;
    if (g.pass.ntiles > 0x7fffffffLL / cluster) return cudaErrorInvalidValue;
    if (a.jq_in) {
        const long long npts = g.pass.lines * ax.n, want = (npts + 1023) / 1024, most = 16LL * current_device_sms();
        err = launch_overlapped(tc_flow_kernel, (unsigned)(want < most || most <= 0 ? want : most), 256, 0, s,
                                g.pass.src, g.pass.dst, npts, g.pass.jin);
        if (err != cudaSuccess) return err;
        g.pass.src = g.pass.dst;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.pass.ntiles * cluster));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)cluster, 1, 1};
    attr[1] = pass_overlap_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, tc_long_kernel<STRIDED>, g);
}

}  // namespace

cudaError_t launch_pass_tc_long(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    return a.inner > 1 ? launch_long<true>(ax, a, s) : launch_long<false>(ax, a, s);
}

}  // namespace sfac
