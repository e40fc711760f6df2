// sfac_tc_pass_f32.cu - FP32 axis passes on the tensor cores: the choice of the tile.
#include "sfac_tc_launch.cuh"

namespace sfac {
namespace {

template <int PARTS>
cudaError_t launch_tc_parts32(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    const long long lines = a.outer * a.inner;
    const int sms = current_device_sms();
    // the narrowest tile with which every SM gets one at most
    if (lines <= 16LL * sms) return launch_tc_axis<float, PARTS, 16>(ax, a, lines, s);
    if (lines <= 32LL * sms) return launch_tc_axis<float, PARTS, 32>(ax, a, lines, s);
    return launch_tc_axis<float, PARTS, 64>(ax, a, lines, s);
}

}  // namespace

cudaError_t launch_pass_tc_f32(const TcAxis& ax, const PassArgs& a, cudaStream_t s) {
    return ax.parts == 2 ? launch_tc_parts32<2>(ax, a, s) : launch_tc_parts32<1>(ax, a, s);
}

}  // namespace sfac
