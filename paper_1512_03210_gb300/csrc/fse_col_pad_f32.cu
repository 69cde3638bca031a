// fse_col_pad_f32.cu -- column-pass instantiations for float: COL_PADF, COL_CROPI.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_col_var<float, COL_PADF>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
template cudaError_t launch_col_var<float, COL_CROPI>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
}  // namespace fse
