// fse_col_plain_f32.cu -- column-pass instantiations for float: COL_FWD, COL_INV.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_col_var<float, COL_FWD>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
template cudaError_t launch_col_var<float, COL_INV>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
}  // namespace fse
