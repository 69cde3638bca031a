// fse_batch_col.cu -- batched column passes (see fse_batch.cu).
#include "fse_batch.cuh"

namespace fse {

template <int N, int VAR, int NP>
__global__ void __launch_bounds__(ColCfg<float, N, VAR, NP>::NT, ColCfg<float, N, VAR, NP>::minb())
k_col_batch(ColArgs a, MulArgs m, const float4* __restrict__ tw, const BatchRun* runs, int kin_full) {
  const BatchRun r = runs[blockIdx.y];
  if constexpr (VAR == COL_KIN2) {
    a.data = r.psi;
    m.kin = kin_full ? r.kin_full : r.kin_half;
  } else {
    a.data = r.spec;
    m.f.a0 = (float)(r.dt * m.scale);
  }
  col_body<float, N, VAR, NP, false>(a, m, tw, blockIdx.x);
}

template <int N, int VAR, int NP>
static cudaError_t colb(const ColArgs& a, const MulArgs& m, long long blocks, const void* tw,
                        const BatchRun* runs, int nr, int kin_full, cudaStream_t st) {
  typedef ColCfg<float, N, VAR, NP> K;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_col_batch<N, VAR, NP>, K::smem(), done);
  if (e != cudaSuccess) return e;
  MulArgs mf = m;
  fill_f32(mf);
  k_col_batch<N, VAR, NP><<<dim3((unsigned)blocks, nr), K::NT, K::smem(), st>>>(
      a, mf, reinterpret_cast<const float4*>(tw), runs, kin_full);
  return cudaGetLastError();
}

template <int VAR>
cudaError_t launch_colb(int n, const ColArgs& a, const MulArgs& m, const void* tw,
                        const BatchRun* runs, int nr, int kin_full, cudaStream_t st) {
  switch (n) {
#define FSE_CASE(n)                                                                                \
  case n:                                                                                          \
    return col_pick<float, n, VAR>(a, nr, [&](auto w, const ColArgs& at, long long blocks) {       \
      return colb<n, VAR, decltype(w)::value>(at, m, blocks, tw, runs, nr, kin_full, st);          \
    });
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_colb<COL_KIN2>(int, const ColArgs&, const MulArgs&, const void*, const BatchRun*,
                                          int, int, cudaStream_t);
template cudaError_t launch_colb<COL_KHAT2>(int, const ColArgs&, const MulArgs&, const void*,
                                           const BatchRun*, int, int, cudaStream_t);

}  // namespace fse
