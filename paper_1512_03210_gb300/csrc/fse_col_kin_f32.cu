// fse_col_kin_f32.cu -- column-pass instantiations for float: COL_KIN, COL_KIN2.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_col_var<float, COL_KIN>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
template cudaError_t launch_col_var<float, COL_KIN2>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
}  // namespace fse
