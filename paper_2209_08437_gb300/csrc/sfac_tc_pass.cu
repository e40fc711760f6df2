// sfac_tc_pass.cu - the FP64 axis pass on the tensor cores (sfac_tc_tile.cuh): one
// launch per pass, persistent CTAs.
#include <atomic>

#include "sfac_tc_tile.cuh"

namespace sfac {
namespace {

struct TcArgs {
    TcPass pass;
    const unsigned char* img;
    unsigned int* status;
    long long wait_cycles;
    int hold;
};

template <int PARTS, int LT, bool STRIDED>
__global__ void __launch_bounds__(TcShape<PARTS, LT>::TOTAL, 1) tc_pass_kernel(const TcArgs g) {
    using Sh = TcShape<PARTS, LT>;
    constexpr int NT = Sh::THREADS;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TcShared sh;
    __shared__ unsigned smax[LT];
    unsigned char* ring = smem + Sh::RING_OFFSET;
    const uint32_t tmem = tc_setup<Sh::COLS, Sh::STAGES>(sh);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    TcState st;
    const int producer = Sh::OWN_PRODUCER ? NT / 32 : 1;
    const int tile_chunks = PARTS * (g.pass.kp >> 5) * kTcSlices;
    if (warp == producer) {
        st.parity = 1;
        st.left = (g.pass.ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x * tile_chunks;
        tc_produce<Sh::STAGES>(sh, st, ring, g.img, tile_chunks, Sh::OWN_PRODUCER ? st.left : Sh::STAGES,
                               g.wait_cycles);
    }
    if (warp < NT / 32) {
        // the test hook: a barrier that nothing completes
        if (g.hold && warp == 0) tc_wait(&sh.never, 0, g.wait_cycles, &sh.abort);
        bool alive = true;
        for (long long tile = blockIdx.x; alive && tile < g.pass.ntiles; tile += gridDim.x)
            alive = tc_tile<PARTS, LT, STRIDED, false, Sh::STAGES>(g.pass, tile, smem, ring, smax, sh, st, tmem, g.img,
                                                                   threadIdx.x, g.wait_cycles);
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

template <int PARTS, int LT, bool STRIDED>
cudaError_t launch_tc(const TcAxis& ax, const PassArgs& a, long long lines, cudaStream_t s) {
    using Sh = TcShape<PARTS, LT>;
    auto kern = tc_pass_kernel<PARTS, LT, STRIDED>;
    static LaunchSetup setup;
    int dev = 0, resident = 0;
    cudaError_t err = set_smem(kern, Sh::SMEM, setup, &dev);
    if (err == cudaSuccess) err = resident_grid(kern, Sh::TOTAL, Sh::SMEM, setup, dev, &resident);
    if (err != cudaSuccess) return err;
    TcArgs g;
    g.pass = tc_pass_of(ax, a);
    g.pass.ntiles = (lines + LT - 1) / LT;
    g.img = static_cast<const unsigned char*>(ax.img);
    g.status = a.status;
    g.wait_cycles = a.wait_cycles;
    g.hold = a.hold;
    if (g.pass.ntiles <= 0) return cudaSuccess;
    const long long grid = g.pass.ntiles < resident ? g.pass.ntiles : resident;
    kern<<<(unsigned)grid, Sh::TOTAL, Sh::SMEM, s>>>(g);
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
    return launch_pass_tc_small(ax, a, s);
}

}  // namespace

cudaError_t launch_pass_tc_f64(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    return ax.parts == 2 ? launch_tc_parts<2>(ax, a, s) : launch_tc_parts<1>(ax, a, s);
}

}  // namespace sfac
