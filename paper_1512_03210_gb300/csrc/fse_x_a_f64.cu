// fse_x_a_f64.cu -- x-pass instantiations for double: XP_A, XP_AL.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_xpass<double, XP_A>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<double, XP_AL>(int, const XArgs&, const void*, const void*, cudaStream_t);
}  // namespace fse
