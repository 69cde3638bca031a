// fse_gs_f32.cu -- ground-state x passes for float.
#define FSE_GSX_INSTANTIATE
#include "fse_gsx.cuh"

namespace fse {
template cudaError_t launch_gs_fwd<float>(int, const GsFwd&, const void*, cudaStream_t);
template cudaError_t launch_gs_inv<float>(int, const GsInv&, const void*, cudaStream_t);
}  // namespace fse
