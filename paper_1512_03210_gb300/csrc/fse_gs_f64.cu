// fse_gs_f64.cu -- ground-state x passes for double.
#define FSE_GSX_INSTANTIATE
#include "fse_gsx.cuh"

namespace fse {
template cudaError_t launch_gs_fwd<double>(int, const GsFwd&, const void*, cudaStream_t);
template cudaError_t launch_gs_inv<double>(int, const GsInv&, const void*, cudaStream_t);
}  // namespace fse
