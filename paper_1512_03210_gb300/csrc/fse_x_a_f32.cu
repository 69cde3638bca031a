// fse_x_a_f32.cu -- x-pass instantiations for float: XP_A, XP_AL.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_xpass<float, XP_A>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<float, XP_AL>(int, const XArgs&, const void*, const void*, cudaStream_t);
}  // namespace fse
