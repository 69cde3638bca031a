// fse_x_e_f32.cu -- x-pass instantiations for float: XP_FWD, XP_INV, XP_E, XP_D.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_xpass<float, XP_FWD>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<float, XP_INV>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<float, XP_E>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<float, XP_D>(int, const XArgs&, const void*, const void*, cudaStream_t);
template int xpass_tiles<float>(int, int);
}  // namespace fse
