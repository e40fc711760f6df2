// sfac_tc_launch.cuh - one launch per axis pass on the tensor cores, persistent
// CTAs (included by the FP64 and the FP32 translation unit).
#pragma once

#include <atomic>

#include "sfac_tc_tile.cuh"
#include "sfac_tc_tile_f32.cuh"

namespace sfac {
namespace {

template <typename R>
constexpr int kSlicesOf = sizeof(R) == 8 ? kTcSlices : kTcSlices32;

template <typename R>
struct TcArgs {
    TcPassT<R> pass;
    const unsigned char* img;
    unsigned int* status;
    long long wait_cycles;
    int hold;
};

template <typename R, int PARTS, int LT, bool STRIDED>
__global__ void __launch_bounds__(TcShape<PARTS, LT, kSlicesOf<R>>::TOTAL, (TcShape<PARTS, LT, kSlicesOf<R>>::CTAS))
tc_pass_kernel(const TcArgs<R> g) {
    using Sh = TcShape<PARTS, LT, kSlicesOf<R>>;
    constexpr int NT = Sh::THREADS;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TcShared sh;
    __shared__ unsigned smax[LT];
    unsigned char* ring = smem + Sh::RING_OFFSET;
    pass_next_may_start();
    const uint32_t tmem = tc_setup<Sh::COLS, Sh::STAGES>(sh);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    TcState st;
    const int producer = Sh::OWN_PRODUCER ? NT / 32 : 1;
    const int stages = PARTS * (g.pass.kp >> 5) * kSlicesOf<R> / Sh::G;  // of the operator
    if (warp == producer) {
        st.parity = 1;
        st.left = (g.pass.ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x * stages;
        tc_produce<Sh::STAGES, Sh::G>(sh, st, ring, g.img, stages, Sh::OWN_PRODUCER ? st.left : Sh::STAGES,
                                      g.wait_cycles, Sh::STAGES);
    }
    if (warp < NT / 32) {
        pass_wait_for_previous();
        // the test hook: a barrier that nothing completes
        if (g.hold && warp == 0) tc_wait(&sh.never, 0, g.wait_cycles, &sh.abort);
        if constexpr (sizeof(R) == 8) {
            tc_tiles<PARTS, LT, STRIDED, Sh::STAGES>(g.pass, smem, ring, smax, sh, st, tmem, g.img, threadIdx.x,
                                                     g.wait_cycles);
        } else {
            bool alive = true;
            for (long long tile = blockIdx.x; alive && tile < g.pass.ntiles; tile += gridDim.x)
                alive = tc_tile_f32<PARTS, LT, STRIDED, Sh::STAGES>(g.pass, tile, smem, ring, smax, sh, st, tmem,
                                                                    g.img, threadIdx.x, g.wait_cycles);
        }
    }
    __syncthreads();
    if (sh.abort) {
        if (warp == producer) tc_drain_copies<Sh::STAGES>(sh, st, g.wait_cycles);
        if (threadIdx.x == 0) {
            mbar_wait_bounded(&sh.done, st.done_parity ^ 1u, g.wait_cycles);
            if (g.status) atomicOr(g.status, SFAC_PASS_TIMEOUT);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, Sh::COLS);
}

template <typename R, int PARTS, int LT, bool STRIDED>
cudaError_t launch_tc(const TcAxis& ax, const PassArgs& a, long long lines, cudaStream_t s) {
    using Sh = TcShape<PARTS, LT, kSlicesOf<R>>;
    auto kern = tc_pass_kernel<R, PARTS, LT, STRIDED>;
    static LaunchSetup setup;
    int dev = 0, resident = 0;
    cudaError_t err = set_smem(kern, Sh::SMEM, setup, &dev);
    if (err == cudaSuccess) err = resident_grid(kern, Sh::TOTAL, Sh::SMEM, setup, dev, &resident);
    if (err != cudaSuccess) return err;
    TcArgs<R> g;
    g.pass = tc_pass_of<R>(ax, a);
    g.pass.ntiles = (lines + LT - 1) / LT;
    g.img = static_cast<const unsigned char*>(ax.img);
    g.status = a.status;
    g.wait_cycles = a.wait_cycles;
    g.hold = a.hold;
    if (g.pass.ntiles <= 0) return cudaSuccess;
    const long long grid = g.pass.ntiles < resident ? g.pass.ntiles : resident;
    // FP64 passes of many rounds keep plain launches: a step of 3D 256^3 (6.7 rounds)
    // took 834 us with overlapped launches and 815 with plain ones, 128^3 (1.7
    // rounds) 111 against 118, and the FP32 step of 255^3 233 against 241.
    if (sizeof(R) == 8 && g.pass.ntiles > 4 * grid) {
        kern<<<(unsigned)grid, Sh::TOTAL, Sh::SMEM, s>>>(g);
        return cudaGetLastError();
    }
    return launch_overlapped(kern, (unsigned)grid, Sh::TOTAL, Sh::SMEM, s, g);
}

template <typename R, int PARTS, int LT>
cudaError_t launch_tc_axis(const TcAxis& ax, const PassArgs& a, long long lines, cudaStream_t s) {
    return a.inner > 1 ? launch_tc<R, PARTS, LT, true>(ax, a, lines, s)
                       : launch_tc<R, PARTS, LT, false>(ax, a, lines, s);
}

}  // namespace
}  // namespace sfac
