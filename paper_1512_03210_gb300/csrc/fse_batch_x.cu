// fse_batch_x.cu -- batched x passes (see fse_batch.cu).
#include "fse_batch.cuh"

namespace fse {

__device__ __forceinline__ double sin_over_dev(double a, double d) {
  const double z = a * d;
  return fabs(z) < 1e-6 ? d * (1.0 - z * z / 6.0) : sin(z) / a;
}

template <int NX, int LN, int KIND>
__global__ void __launch_bounds__(XCfg<float, NX, LN>::NT, XCfg<float, NX, LN>::minb())
k_xpass_batch(XArgs a, const float4* __restrict__ twn, const float4* __restrict__ tw2n,
              const BatchRun* runs, const double* t0p, int step) {
  const BatchRun r = runs[blockIdx.y];
  a.psi = r.psi;
  a.spec = a.use_spec ? r.spec : nullptr;
  if constexpr (KIND == XP_A) {
    // exact time integral of the rotating harmonic trap over the run's step
    // (Eq. int_poten); the call's start time t0 is a device scalar, so that a
    // captured graph of the step sequence serves every call. One thread
    // evaluates the float64 sines and cosines (GB300's float64 pipe is
    // narrow) and the block reads the coefficients from shared memory.
    __shared__ double trap[3];
    if (threadIdx.x == 0) {
      const double ta = *t0p + step * r.dt, d = r.dt, mid = 2.0 * ta + d;
      const double C2 = cos(r.omega * mid) * sin_over_dev(r.omega, d);
      const double S2 = sin(r.omega * mid) * sin_over_dev(r.omega, d);
      trap[0] = 0.25 * (r.gx2 * (d + C2) + r.gy2 * (d - C2));
      trap[1] = 0.25 * (r.gx2 * (d - C2) + r.gy2 * (d + C2));
      trap[2] = 0.5 * (r.gx2 - r.gy2) * S2;
    }
    __syncthreads();
    a.pa = trap[0];
    a.pb = trap[1];
    a.pc = trap[2];
    a.pe = 0.0;
    a.beta_dt = r.beta * r.dt;
    a.lam = r.lam;
    fill_f32_phase(a);
  }
  xpass_body<float, NX, LN, KIND, false>(a, twn, tw2n, blockIdx.x);
}

template <int NX, int LN, int KIND>
static cudaError_t xb(const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                      const double* t0, int step, cudaStream_t st) {
  typedef XCfg<float, NX, LN> K;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_xpass_batch<NX, LN, KIND>, K::smem(), done);
  if (e != cudaSuccess) return e;
  dim3 grid((a.nlines + LN - 1) / LN, nr);
  XArgs af = a;
  fill_f32(af);
  k_xpass_batch<NX, LN, KIND><<<grid, K::NT, K::smem(), st>>>(af, reinterpret_cast<const float4*>(twn),
                                                              reinterpret_cast<const float4*>(tw2n), runs, t0, step);
  return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_xb_kind(int nx, const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                                  const double* t0, int step, cudaStream_t st) {
  switch (nx) {
#define FSE_CASE(n)                                                                                          \
  case n:                                                                                                    \
    return xpass_pick<float, n>(a.nlines, nr) == XWidths<float, n>::wide()                                   \
               ? xb<n, XWidths<float, n>::wide(), KIND>(a, twn, tw2n, runs, nr, t0, step, st)                \
               : xb<n, XWidths<float, n>::narrow(), KIND>(a, twn, tw2n, runs, nr, t0, step, st);
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_xb(int kind, int nx, const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                      const double* t0, int step, cudaStream_t st) {
  switch (kind) {
    case XP_FWD: return launch_xb_kind<XP_FWD>(nx, a, twn, tw2n, runs, nr, t0, step, st);
    case XP_INV: return launch_xb_kind<XP_INV>(nx, a, twn, tw2n, runs, nr, t0, step, st);
    case XP_E: return launch_xb_kind<XP_E>(nx, a, twn, tw2n, runs, nr, t0, step, st);
    default: return launch_xb_kind<XP_A>(nx, a, twn, tw2n, runs, nr, t0, step, st);
  }
}

}  // namespace fse
