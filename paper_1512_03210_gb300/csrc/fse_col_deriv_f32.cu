// fse_col_deriv_f32.cu -- column-pass instantiations for float: COL_RMUL, COL_DY, COL_LZ.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_col_var<float, COL_RMUL>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
template cudaError_t launch_col_var<float, COL_DY>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
template cudaError_t launch_col_var<float, COL_LZ>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
}  // namespace fse
