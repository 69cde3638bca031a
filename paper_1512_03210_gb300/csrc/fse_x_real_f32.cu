// fse_x_real_f32.cu -- x-pass instantiations for float: XP_R, XP_LZ.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_xpass<float, XP_R>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<float, XP_LZ>(int, const XArgs&, const void*, const void*, cudaStream_t);
}  // namespace fse
