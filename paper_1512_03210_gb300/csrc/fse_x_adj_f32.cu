// fse_x_adj_f32.cu -- x-pass instantiations for float: XP_ADJ1, XP_ADJ2.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_xpass<float, XP_ADJ1>(int, const XArgs&, const void*, const void*, cudaStream_t);
template cudaError_t launch_xpass<float, XP_ADJ2>(int, const XArgs&, const void*, const void*, cudaStream_t);
}  // namespace fse
