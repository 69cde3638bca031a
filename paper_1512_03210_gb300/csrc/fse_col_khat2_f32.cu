// fse_col_khat2_f32.cu -- column-pass instantiations for float: COL_KHAT2.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_col_var<float, COL_KHAT2>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
}  // namespace fse
