// sfac_tc_pass.cu - FP64 axis passes on the tensor cores: the choice of the tile.
#include "sfac_tc_launch.cuh"

namespace sfac {
namespace {

template <int PARTS>
cudaError_t launch_tc_parts(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    const long long lines = a.outer * a.inner;
    const int sms = current_device_sms();
    // The narrowest tile with which every SM gets one at most: a tile's time is
    // mostly latency until it is 64 lines wide, so two rounds of narrow tiles lose to
    // one round of tiles twice as wide.
    if (lines <= 8LL * sms) return launch_pass_tc_small(ax, a, s);
    if (lines <= 16LL * sms) return launch_tc_axis<double, PARTS, 16>(ax, a, lines, s);
    if (lines <= 32LL * sms) return launch_tc_axis<double, PARTS, 32>(ax, a, lines, s);
    return launch_tc_axis<double, PARTS, 64>(ax, a, lines, s);
}

}  // namespace

cudaError_t launch_pass_tc_f64(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    if (ax.n > kTcMaxN) return launch_pass_tc_long(ax, a, s);
    return ax.parts == 2 ? launch_tc_parts<2>(ax, a, s) : launch_tc_parts<1>(ax, a, s);
}

}  // namespace sfac
