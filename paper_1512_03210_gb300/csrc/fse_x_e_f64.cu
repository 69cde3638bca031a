// fse_x_e_f64.cu -- x-pass instantiations for double: XP_FWD, XP_INV, XP_E, XP_D.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_xpass<double, XP_FWD>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<double, XP_INV>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<double, XP_E>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<double, XP_D>(int, const XArgs&, const void*, const void*, cudaStream_t);
template int xpass_tiles<double>(int, int);
}  // namespace fse
