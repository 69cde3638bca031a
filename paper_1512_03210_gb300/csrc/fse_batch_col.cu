// fse_batch_col.cu -- batched column passes (see fse_batch.cu).
#include "fse_batch.cuh"

namespace fse {

__device__ double sin_over_dev(double a, double d) {
  const double z = a * d;
  return fabs(z) < 1e-6 ? d * (1.0 - z * z / 6.0) : sin(z) / a;
}

// Exact time integral of the rotating harmonic trap over step `step` of a run
// (Eq. int_poten); the call's start time is a device scalar, so that a captured
// graph of the step sequence serves every call.
__device__ __forceinline__ float4 batch_trap(const BatchRun& r, double t0, int step) {
  const double ta = t0 + step * r.dt, d = r.dt, mid = 2.0 * ta + d;
  const double C2 = cos(r.omega * mid) * sin_over_dev(r.omega, d);
  const double S2 = sin(r.omega * mid) * sin_over_dev(r.omega, d);
  return make_float4((float)(0.25 * (r.gx2 * (d + C2) + r.gy2 * (d - C2))),
                     (float)(0.25 * (r.gx2 * (d - C2) + r.gy2 * (d + C2))), (float)(0.5 * (r.gx2 - r.gy2) * S2), 0.f);
}

// The trap's float64 sines and cosines, one block per run and one thread per
// step, ahead of the steps that read them: at the head of every block of the
// phase pass they were 27 of its 156 us at 57 runs of 512^2 (the FP64 pipe), and
// in an extra block of the kinetic pass they cost that pass 13 us.
__global__ void __launch_bounds__(kTrapSteps) k_batch_trap(const BatchRun* runs, const double* t0, int step0, int nsteps,
                                                           float4* trap) {
  const int n = threadIdx.x;
  if (n < nsteps) trap[(size_t)n * gridDim.x + blockIdx.x] = batch_trap(runs[blockIdx.x], *t0, step0 + n);
}
cudaError_t launch_batch_trap(const BatchRun* runs, int nr, const double* t0, int step0, int nsteps, float4* trap,
                              cudaStream_t st) {
  k_batch_trap<<<nr, kTrapSteps, 0, st>>>(runs, t0, step0, nsteps, trap);
  return cudaGetLastError();
}

template <int N, int VAR, int NP>
__global__ void __launch_bounds__(ColCfg<float, N, VAR, NP>::NT, ColCfg<float, N, VAR, NP>::minb())
k_col_batch(ColArgs a, MulArgs m, const float4* __restrict__ tw, const BatchRun* runs, int kin_full) {
  const BatchRun r = runs[blockIdx.y];
  if constexpr (VAR == COL_KIN2) {
    a.data = r.psi;
    m.kin = kin_full ? r.kin_full : r.kin_half;
  } else {
    a.data = r.spec;
    m.f.a0 = r.a0;
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
