// fse_batch_x.cu -- batched x passes (see fse_batch.cu).
#include "fse_batch.cuh"

namespace fse {

template <int NX, int LN, int KIND>
__global__ void __launch_bounds__(XCfg<float, NX, LN>::NT, XCfg<float, NX, LN>::minb())
k_xpass_batch(XArgs a, const float4* __restrict__ twn, const float4* __restrict__ tw2n,
              const BatchRun* runs, const float4* trap) {
  const BatchRun r = runs[blockIdx.y];
  a.psi = r.psi;
  a.spec = a.use_spec ? r.spec : nullptr;
  if constexpr (KIND == XP_A) {
    const float4 t = trap[blockIdx.y];
    a.f.pa = t.x;
    a.f.pb = t.y;
    a.f.pc = t.z;
    a.f.pe = 0.f;
    a.f.beta_dt = r.beta_dt;
    a.f.lam = r.lam;
  }
  xpass_body<float, NX, LN, KIND, false>(a, twn, tw2n, blockIdx.x);
}

template <int NX, int LN, int KIND>
static cudaError_t xb(const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                      const float4* trap, cudaStream_t st) {
  typedef XCfg<float, NX, LN> K;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_xpass_batch<NX, LN, KIND>, K::smem(), done);
  if (e != cudaSuccess) return e;
  dim3 grid((a.nlines + LN - 1) / LN, nr);
  XArgs af = a;
  fill_f32(af);
  k_xpass_batch<NX, LN, KIND><<<grid, K::NT, K::smem(), st>>>(af, reinterpret_cast<const float4*>(twn),
                                                              reinterpret_cast<const float4*>(tw2n), runs, trap);
  return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_xb_kind(int nx, const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                                  const float4* trap, cudaStream_t st) {
  switch (nx) {
#define FSE_CASE(n)                                                                                          \
  case n:                                                                                                    \
    return xpass_pick<float, n>(a.nlines, nr) == XWidths<float, n>::wide()                                   \
               ? xb<n, XWidths<float, n>::wide(), KIND>(a, twn, tw2n, runs, nr, trap, st)                \
               : xb<n, XWidths<float, n>::narrow(), KIND>(a, twn, tw2n, runs, nr, trap, st);
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_xb(int kind, int nx, const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                      const float4* trap, cudaStream_t st) {
  switch (kind) {
    case XP_FWD: return launch_xb_kind<XP_FWD>(nx, a, twn, tw2n, runs, nr, trap, st);
    case XP_INV: return launch_xb_kind<XP_INV>(nx, a, twn, tw2n, runs, nr, trap, st);
    case XP_E: return launch_xb_kind<XP_E>(nx, a, twn, tw2n, runs, nr, trap, st);
    default: return launch_xb_kind<XP_A>(nx, a, twn, tw2n, runs, nr, trap, st);
  }
}

}  // namespace fse
