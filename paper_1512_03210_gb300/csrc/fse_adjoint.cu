// fse_adjoint.cu -- transpose of one split step (gradients; the paper has no adjoint).
//
// Forward step (Section 4.2, Eqs. tssp1-tssp3): u1 = K psi_n, rho = |u1|^2,
// Theta = dt beta rho + lambda Kc rho + P(gamma), u2 = u1 exp(-i Theta),
// psi_{n+1} = K u2, with K the kinetic half step and Kc the padded
// convolution with the time-integrated kernel (real, even multiplier, so Kc
// is symmetric). Cotangents are g = dJ/dRe + i dJ/dIm. Pulling g back:
//   g_u2 = K^H g                                    (conjugate kinetic phase)
//   h    = exp(+i Theta) g_u2,  r = Im(conj(g_u2) u2) = Im(conj(h) u1)
//   g_u1 = h + 2 (dt beta r + lambda Kc r) u1
//   g_n  = K^H g_u1
//   dJ/dgamma_v = sum_x r dP/dgamma_v
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fse.h"
#include "fse_internal.h"
#include "fse_passes.cuh"

namespace fse {

constexpr long long kAdjStride = 65536;  // partials per gradient slot
constexpr long long kAdjBase = 0;         // slots 0..2 of the reduction region (shared with observables)
constexpr long long kAdjOut = 16LL * 65536 + 8;   // scalar results
constexpr long long kAdjSums = 14LL * 65536;       // a sweep's sums, after its partials

// out[b] = sum of the count partials of group b (fixed order)
__global__ void __launch_bounds__(256) k_sum_groups(const double* part, int count, long long stride, double* out) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += part[blockIdx.x * stride + i];
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) out[blockIdx.x] = acc;
}

// Scalars of the two adjoint x passes of the step [ta, tb] with trap frequencies gamma.
XArgs adjoint_args(fse_plan* P, void* g, void* spec, const void* u1, double ta, double tb, const double* gamma) {
  double pc[4];
  trap_coefficients(P, ta, tb, gamma, pc);
  XArgs x = x_args(P, g, spec);
  x.aux = u1;
  x.ix0 = origin_index(P, 0);
  x.beta_dt = P->p.beta * P->p.dt;
  x.lam = P->p.lambda;
  x.pa = pc[0];
  x.pb = pc[1];
  x.pc = pc[2];
  x.pe = pc[3];
  lattice_nodes(P, ta, tb, x);
  // dP/dgamma_v = gamma_v * int (A x~)_v^2 dtau: unit-frequency trap integrals times 2 gamma_v
  for (int v = 0; v < 3; ++v) {
    double one[3] = {0.0, 0.0, 0.0};
    one[v] = 1.0;
    double c[4] = {0, 0, 0, 0};
    if (v < P->dim) trap_coefficients(P, ta, tb, one, c);  // 1/2 int (A x~)_v^2 dtau
    const double gv = v < P->dim ? (gamma ? gamma[v] : P->p.gamma[v]) : 0.0;
    for (int k = 0; k < 4; ++k) x.dp[4 * v + k] = 2.0 * gv * c[k];
  }
  return x;
}

// K or K^H on a physical field: fwd x, y/z passes with the phase, inv x.
fse_status kinetic_full(fse_plan* P, void* f, double sign) {
  XArgs xa = x_args(P, f, nullptr);
  fse_status st;
  if ((st = xpass(P, XP_FWD, xa)) != FSE_OK) return st;
  if ((st = kinetic_yz(P, f, sign, P->p.dt)) != FSE_OK) return st;
  return xpass(P, XP_INV, xa);
}

}  // namespace fse

using namespace fse;

extern "C" fse_status fse_step_adjoint(fse_plan_t P, const void* psi_n, void* g, double t_n,
                                       const double* gamma_n, double* dgamma_n) {
  if (!P || !psi_n || !g) return FSE_ERR_INVALID;
  if (!P->ws || !P->precomputed) return fail(P, FSE_ERR_INVALID, "fse_kernel_precompute has not run");
  if (P->p.renormalize) return fail(P, FSE_ERR_UNSUPPORTED, "adjoint of a renormalised plan");
  if (P->p.order != 2) return fail(P, FSE_ERR_UNSUPPORTED, "adjoint of the fourth-order composition");
  if (reinterpret_cast<uintptr_t>(g) % P->csize != 0 || reinterpret_cast<uintptr_t>(psi_n) % P->csize != 0)
    return fail(P, FSE_ERR_INVALID, "misaligned buffer");
  const double dt = P->p.dt, ta = t_n, tb = t_n + dt;
  void* u1 = P->ws_ptr(P->off_tmp);
  void* spec = P->ws_ptr(P->off_spec);
  double* red = reinterpret_cast<double*>(P->ws_ptr(P->off_red));
  const bool nl = has_nonlocal(P);
  fse_status st;
  cudaError_t e;

  // u1 = K psi_n and (with a nonlocal term) the x-half-spectrum of rho = |u1|^2
  XArgs xu = x_args(P, u1, nl ? spec : nullptr);
  xu.aux = psi_n;
  if ((st = xpass(P, XP_FWD, xu)) != FSE_OK) return st;
  xu.aux = nullptr;
  if ((st = kinetic_yz(P, u1, 1.0, dt)) != FSE_OK) return st;
  if (nl) {
    if ((st = xpass(P, XP_E, xu)) != FSE_OK) return st;
    if ((st = nonlocal_yz(P, spec, ta, tb, true, nullptr, 1.0)) != FSE_OK) return st;
  } else {
    if ((st = xpass(P, XP_INV, xu)) != FSE_OK) return st;
  }
  // g_u2 = K^H g
  if ((st = kinetic_full(P, g, -1.0)) != FSE_OK) return st;

  // pass 1: h, r (and its spectrum), trap-gradient partials
  XArgs x1 = adjoint_args(P, g, nl ? spec : nullptr, u1, ta, tb, gamma_n);
  x1.part = dgamma_n ? red + kAdjBase : nullptr;
  x1.part_stride = kAdjStride;
  const int xblocks = x_tiles(P, x1.nlines);
  if (dgamma_n && xblocks > kAdjStride) return fail(P, FSE_ERR_UNSUPPORTED, "adjoint: grid too large");
  if ((st = xpass(P, XP_ADJ1, x1)) != FSE_OK) return st;
  // Kc r, then pass 2: g_u1 = h + 2 q u1
  if (nl && (st = nonlocal_yz(P, spec, ta, tb, true, nullptr, 1.0)) != FSE_OK) return st;
  XArgs x2 = x1;
  x2.part = nullptr;
  if ((st = xpass(P, XP_ADJ2, x2)) != FSE_OK) return st;
  // g_n = K^H g_u1
  if ((st = kinetic_full(P, g, -1.0)) != FSE_OK) return st;

  if (dgamma_n) {
    double* out = red + kAdjOut;
    k_sum_groups<<<3, 256, 0, P->stream>>>(red + kAdjBase, xblocks, kAdjStride, out);
    if ((st = launched(P, cudaGetLastError(), "adjoint gradient sum")) != FSE_OK) return st;
    double h3[3];
    if ((e = cudaMemcpyAsync(h3, out, sizeof(h3), cudaMemcpyDeviceToHost, P->stream)) != cudaSuccess)
      return cuda_fail(P, e, "adjoint read");
    if ((e = cudaStreamSynchronize(P->stream)) != cudaSuccess) return cuda_fail(P, e, "adjoint sync");
    for (int v = 0; v < P->dim; ++v) dgamma_n[v] = h3[v];
  }
  return FSE_OK;
}

extern "C" fse_status fse_adjoint_sweep(fse_plan_t P, const void* psi_0, void* states, void* g, double t0, int nsteps,
                                        const double* gamma_per_step, double* dgamma) {
  if (!P || !psi_0 || !states || !g || nsteps < 1) return FSE_ERR_INVALID;
  if (!P->ws || !P->precomputed) return fail(P, FSE_ERR_INVALID, "fse_kernel_precompute has not run");
  if (P->p.renormalize) return fail(P, FSE_ERR_UNSUPPORTED, "adjoint of a renormalised step");
  if (P->p.order != 2) return fail(P, FSE_ERR_UNSUPPORTED, "adjoint of the fourth-order composition");
  if (reinterpret_cast<uintptr_t>(g) % P->csize != 0 || reinterpret_cast<uintptr_t>(psi_0) % P->csize != 0 ||
      reinterpret_cast<uintptr_t>(states) % P->csize != 0)
    return fail(P, FSE_ERR_INVALID, "misaligned buffer");
  const double dt = P->p.dt;
  void* w = P->ws_ptr(P->off_tmp);
  const bool nl = has_nonlocal(P);
  void* spec = nl ? P->ws_ptr(P->off_spec) : nullptr;
  double* red = reinterpret_cast<double*>(P->ws_ptr(P->off_red));
  const int lines = P->ny * (P->dim == 3 ? P->nz : 1), tiles = x_tiles(P, lines), dim = P->dim;
  // the trap-gradient partials of as many steps as fit are summed together
  const int batch = (int)std::min<long long>(kAdjSums / 3 / tiles, 512);
  if (dgamma && batch < 1) return fail(P, FSE_ERR_UNSUPPORTED, "adjoint: grid too large");
  auto state = [&](int k) { return static_cast<char*>(states) + (size_t)k * P->psi_bytes; };
  auto gam = [&](int k) { return gamma_per_step ? gamma_per_step + (size_t)k * dim : nullptr; };
  fse_status st;

  // forward: u1 of every step into states (the field itself, x-spectral between
  // the steps, in the scratch field); the last step's potential stays in S
  XArgs xw = x_args(P, w, spec);
  xw.aux = psi_0;
  if ((st = xpass(P, XP_FWD, xw)) != FSE_OK) return st;
  for (int k = 0; k < nsteps; ++k) {
    const double ta = t0 + k * dt, tb = t0 + (k + 1) * dt;
    if ((st = kinetic_yz(P, w, k == 0 ? 1.0 : 2.0, dt)) != FSE_OK) return st;
    XArgs xe = x_args(P, w, spec);
    xe.out = state(k);
    if ((st = xpass(P, nl ? XP_E : XP_INV, xe)) != FSE_OK) return st;
    if (nl && (st = nonlocal_yz(P, spec, ta, tb, true, nullptr, 1.0)) != FSE_OK) return st;
    if (k + 1 == nsteps) break;
    XArgs xA = adjoint_args(P, w, spec, state(k), ta, tb, gam(k));
    if ((st = xpass(P, P->p.lat_amp != 0.0 ? XP_AL : XP_A, xA)) != FSE_OK) return st;
  }
  // backward: K^H of the end of one step and the start of the one before merge
  XArgs xg = x_args(P, g, nullptr);
  if ((st = xpass(P, XP_FWD, xg)) != FSE_OK) return st;
  std::vector<double> host(dgamma ? 3 * (size_t)batch : 0);
  int held = 0;  // steps whose partials wait
  for (int k = nsteps - 1; k >= 0; --k) {
    const double ta = t0 + k * dt, tb = t0 + (k + 1) * dt;
    if ((st = kinetic_yz(P, g, k + 1 == nsteps ? -1.0 : -2.0, dt)) != FSE_OK) return st;
    if ((st = xpass(P, XP_INV, xg)) != FSE_OK) return st;
    if (nl && k + 1 != nsteps) {
      XArgs xd = x_args(P, state(k), spec);
      if ((st = xpass(P, XP_D, xd)) != FSE_OK) return st;
      if ((st = nonlocal_yz(P, spec, ta, tb, true, nullptr, 1.0)) != FSE_OK) return st;
    }
    XArgs x1 = adjoint_args(P, g, spec, state(k), ta, tb, gam(k));
    XArgs x2 = x1;
    x1.part = dgamma ? red + 3LL * held * tiles : nullptr;
    x1.part_stride = tiles;
    if ((st = xpass(P, XP_ADJ1, x1)) != FSE_OK) return st;
    if (nl && (st = nonlocal_yz(P, spec, ta, tb, true, nullptr, 1.0)) != FSE_OK) return st;
    if ((st = xpass(P, XP_ADJ2, x2)) != FSE_OK) return st;
    if ((st = xpass(P, XP_FWD, xg)) != FSE_OK) return st;
    if (dgamma && (++held == batch || k == 0)) {
      double* out = red + kAdjSums;
      k_sum_groups<<<3 * held, 256, 0, P->stream>>>(red, tiles, tiles, out);
      if ((st = launched(P, cudaGetLastError(), "adjoint gradient sum")) != FSE_OK) return st;
      cudaError_t e = cudaMemcpyAsync(host.data(), out, sizeof(double) * 3 * held, cudaMemcpyDeviceToHost, P->stream);
      if (e != cudaSuccess) return cuda_fail(P, e, "adjoint read");
      if (k > 0) {
        if ((e = cudaStreamSynchronize(P->stream)) != cudaSuccess) return cuda_fail(P, e, "adjoint sync");
        for (int i = 0; i < held; ++i)
          for (int v = 0; v < dim; ++v) dgamma[(size_t)(k + held - 1 - i) * dim + v] = host[3 * i + v];
        held = 0;
      }
    }
  }
  if ((st = kinetic_yz(P, g, -1.0, dt)) != FSE_OK) return st;
  if ((st = xpass(P, XP_INV, xg)) != FSE_OK) return st;
  cudaError_t e = cudaStreamSynchronize(P->stream);
  if (e != cudaSuccess) return cuda_fail(P, e, "adjoint sync");
  for (int i = 0; i < held; ++i)
    for (int v = 0; v < dim; ++v) dgamma[(size_t)(held - 1 - i) * dim + v] = host[3 * i + v];
  return FSE_OK;
}
