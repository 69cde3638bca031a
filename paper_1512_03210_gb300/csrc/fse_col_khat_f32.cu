// fse_col_khat_f32.cu -- column-pass instantiations for float: COL_KHAT.
#include "fse_launch.cuh"

namespace fse {
template cudaError_t launch_col_var<float, COL_KHAT>(int, const ColArgs&, const MulArgs&, const void*, cudaStream_t);
}  // namespace fse
