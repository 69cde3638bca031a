// fse_observables.cu -- float64 observables on the device (Section 1, Eqs. mass, energy;
// Section 4.1, Eqs. AME, CoM, ConWidth).
//
// phi lives in the rotating Lagrangian frame at time t. The energy is that of
// Eq. SFSE (rotation term included); the kinetic term, the interactions and
// L_z are invariant under the frame rotation and V(A(t) x~) = W(x~, t), so
// every term is evaluated in x~. Centre of mass and widths are returned in
// the frame of Eq. SFSE, x = A(t) x~.
//
// Reductions: each block accumulates in float64 and writes one partial per
// slot; one block per slot then sums the partials in a fixed order, so the
// result does not depend on scheduling.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "fse.h"
#include "fse_internal.h"
#include "fse_passes.cuh"

namespace fse {

enum {
  SL_MASS = 0, SL_RHO2, SL_WRHO, SL_X, SL_Y, SL_Z, SL_XX, SL_YY, SL_ZZ, SL_XY,
  SL_KIN, SL_LZY, SL_LZX, SL_NON, NSLOT
};
constexpr int kPartStride = 65536;  // partials per slot (>= x-pass blocks of the largest grid)
constexpr int kRedBlocks = 1024;

struct ObsArgs {
  int nx, ny, nlines;
  double lo[3], h[3];
  double c, s;   // cos, sin of Omega t
  double lat_amp, lat_k[3];  // optical lattice lat_amp sum_v sin^2(lat_k[v] x_v)
  int ic[3];     // the moments' origin: the grid index next to the coordinates' zero
  bool by_points;  // the x, y part of the harmonic trap energy point by point
  double g2[3];  // gamma_v^2 / 2
};

// CW points of a line 32 apart (zero past the end)
template <typename Real>
__device__ __forceinline__ Vec<typename LaneOf<Real>::T> pair_at(const typename Cplx<Real>::T* row, int x, int nx) {
  constexpr int CW = sizeof(typename LaneOf<Real>::T) / sizeof(Real);
  Real re[CW], im[CW];
#pragma unroll
  for (int q = 0; q < CW; ++q) {
    const bool in = x + 32 * q < nx;
    re[q] = in ? row[x + 32 * q].x : Real(0);
    im[q] = in ? row[x + 32 * q].y : Real(0);
  }
  return {lane_of(re), lane_of(im)};
}

// energies of a lane's points of a line that are formed in float64 point by
// point: the lattice's and (by_points) the harmonic trap's along x and y
template <typename C> __device__ __forceinline__ double potential_line(const C* row, const ObsArgs& o, int iy, int iz, int lane) {
  const double y = o.lo[1] + o.h[1] * iy, z = o.lo[2] + o.h[2] * iz;
  double acc = 0.0;
  for (int x = lane; x < o.nx; x += 32) {
    const C u = row[x];
    const double rho = (double)u.x * u.x + (double)u.y * u.y, xx = o.lo[0] + o.h[0] * x;
    const double X = o.c * xx + o.s * y, Y = -o.s * xx + o.c * y;
    double w = 0.0;
    if (o.by_points) w = o.g2[0] * X * X + o.g2[1] * Y * Y;
    if (o.lat_amp != 0.0) {
      const double sx = sin(o.lat_k[0] * X), sy = sin(o.lat_k[1] * Y), sz = sin(o.lat_k[2] * z);
      w += o.lat_amp * (sx * sx + sy * sy + sz * sz);
    }
    acc += w * rho;
  }
  return acc;
}

// Moments of the density, one warp per line, in index units from the index next
// to the coordinates' zero: along a line only the sums of rho, rho^2, rho i and
// rho i^2 are formed, and a line's y and z enter once; the coordinates and the
// harmonic trap energy follow from the sums on the host. From that origin the
// terms of x = c + h i and x^2 = c^2 + 2 c h i + h^2 i^2 have one sign, or c is
// within half a spacing of zero (their moduli then add up to nine times x^2 at
// most). From the grid's middle they cancel in a box to one side of zero: x^2
// of a cloud at 0.5 in [0, 16] was 5e-14 off, now 1e-16. In float64 that is about 11
// slots of the FP64 pipe per point in place of 45 (128^3 float32 fields: 172 ->
// 56 us, the pipe's time); float fields are summed by three floats (ExactSum):
// 33 us, the chains of two-sums of the 16 warps that 126 registers leave an SM.
// Slots: rho, rho^2, point energies, and rho times i, j, k, i i, j j, k k, i j.
__global__ void __launch_bounds__(256) k_obs_phys(const float2* __restrict__ psi, ObsArgs o, double* part) {
  __shared__ double red[10 * 256];
  typedef ExactSum<float2> Sum;
  const int lane = threadIdx.x & 31, nw = gridDim.x * 8;
  Sum t0, t1, ti, tj, tk, tii, tjj, tkk, tij;
  double lat = 0.0;
  RunScale<float2> su;
  for (int l = blockIdx.x * 8 + (threadIdx.x >> 5); l < o.nlines; l += nw) {
    const float2* row = psi + (long long)l * o.nx;
    const int iy = l % o.ny, iz = l / o.ny;
    float um = 0.f;
#pragma unroll 2
    for (int x = lane; x < o.nx; x += 64) {
      const Vec<float2> u = pair_at<float>(row, x, o.nx);
      um = lmax_abs(lmax_abs(um, u.re), u.im);
    }
    su.grow(um, [&](float2 r) {
      const float2 r2 = lmul(r, r);
      t0.rescale(r2), ti.rescale(r2), tj.rescale(r2), tk.rescale(r2), tii.rescale(r2), tjj.rescale(r2);
      tkk.rescale(r2), tij.rescale(r2), t1.rescale(lmul(r2, r2));
    });
    Sum s0, s1;
#pragma unroll 2
    for (int x = lane; x < o.nx; x += 64) {
      const Vec<float2> u = pair_at<float>(row, x, o.nx);
      const Sum rho = Sum::density(lmul(su.scale, u.re), lmul(su.scale, u.im));
      const float i = (float)(x - o.ic[0]);
      const float2 i2 = make_float2(i, i + 32.f);
      s0.add(rho);
      s1.prod(i2, rho);
      tii.prod(lmul(i2, i2), rho);
      t1.square(rho);
    }
    if (o.by_points || o.lat_amp != 0.0) lat += potential_line(row, o, iy, iz, lane);
    const float j = (float)(iy - o.ic[1]), k = (float)(iz - o.ic[2]);
    const float2 j2 = make_float2(j, j), k2 = make_float2(k, k);
    t0.add(s0);
    ti.add(s1);
    tj.prod(j2, s0);
    tk.prod(k2, s0);
    tjj.prod(lmul(j2, j2), s0);
    tkk.prod(lmul(k2, k2), s0);
    tij.prod(j2, s1);
  }
  const double v2 = su.inv * su.inv;
  auto val = [&](const Sum& s) { return v2 * (s.get(0) + s.get(1)); };
  const double acc[10] = {val(t0), v2 * val(t1), lat, val(ti), val(tj), val(tk), val(tii), val(tjj), val(tkk), val(tij)};
  block_sums(acc, red, [&](int k, double v) { part[k * kPartStride + blockIdx.x] = v; });
}

__global__ void __launch_bounds__(256) k_obs_phys(const double2* __restrict__ psi, ObsArgs o, double* part) {
  __shared__ double red[10 * 256];
  const int lane = threadIdx.x & 31, nw = gridDim.x * 8;
  double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int l = blockIdx.x * 8 + (threadIdx.x >> 5); l < o.nlines; l += nw) {
    const double2* row = psi + (long long)l * o.nx;
    const int iy = l % o.ny, iz = l / o.ny;
    double s0 = 0.0, s1 = 0.0, i0 = lane - o.ic[0];
#pragma unroll 4
    for (int x = lane; x < o.nx; x += 32, i0 += 32.0) {
      const double2 u = row[x];
      const double rho = u.x * u.x + u.y * u.y, t = rho * i0;
      s0 += rho;
      acc[1] = fma(rho, rho, acc[1]);
      s1 += t;
      acc[6] = fma(t, i0, acc[6]);
    }
    if (o.by_points || o.lat_amp != 0.0) acc[2] += potential_line(row, o, iy, iz, lane);
    const double j = iy - o.ic[1], k = iz - o.ic[2], a = j * s0, b = k * s0;
    acc[0] += s0;
    acc[3] += s1;
    acc[4] += a;
    acc[5] += b;
    acc[7] = fma(j, a, acc[7]);
    acc[8] = fma(k, b, acc[8]);
    acc[9] = fma(j, s1, acc[9]);
  }
  block_sums(acc, red, [&](int k, double v) { part[k * kPartStride + blockIdx.x] = v; });
}

// sum over the spectrum of (|k|^2 + m^2)^s |phi^_k|^2 (unnormalised DFT), one warp per line
template <typename Real>
__global__ void __launch_bounds__(256) k_obs_kin(const typename Cplx<Real>::T* __restrict__ sp, ObsArgs o, int nz,
                                                 double dkx, double dky, double dkz, double s, double m2,
                                                 double* part) {
  __shared__ double red[32];
  const int lane = threadIdx.x & 31, nw = gridDim.x * 8;
  typedef typename LaneOf<Real>::T L;
  constexpr int CW = sizeof(L) / sizeof(Real);
  ExactSum<L> sum;
  RunScale<L> su;
  // the weights grow with |k|: their scale is the corner's
  const Real cx = Real(dkx) * Real(o.nx / 2), cy = Real(dky) * Real(o.ny / 2), cz = Real(dkz) * Real(nz / 2);
  const Pow2<L> sw = pow2_scale<L>((float)pow(cx * cx + cy * cy + cz * cz + Real(m2), Real(s)));
  for (int l = blockIdx.x * 8 + (threadIdx.x >> 5); l < o.nlines; l += nw) {
    const typename Cplx<Real>::T* row = sp + (long long)l * o.nx;
    const Real ky = Real(dky) * Real(wrap_index(l % o.ny, o.ny));
    const Real kz = nz > 1 ? Real(dkz) * Real(wrap_index(l / o.ny, nz)) : Real(0);
    auto at = [&](int x) { return pair_at<Real>(row, x, o.nx); };
    float um = 0.f;
    if constexpr (sizeof(Real) == 4) {
#pragma unroll 2
      for (int x = lane; x < o.nx; x += 64) {
        const Vec<L> u = at(x);
        um = lmax_abs(lmax_abs(um, u.re), u.im);
      }
    }
    su.grow(um, [&](L r) { sum.rescale(lmul(r, r)); });
#pragma unroll 2
    for (int x = lane; x < o.nx; x += 32 * CW) {
      Real w[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) {
        const Real kx = Real(dkx) * Real(wrap_index(x + 32 * q, o.nx));
        w[q] = x + 32 * q < o.nx ? pow(kx * kx + ky * ky + kz * kz + Real(m2), Real(s)) : Real(0);
      }
      const Vec<L> u = at(x);
      sum.dens(lmul(sw.scale, lane_of(w)), lmul(su.scale, u.re), lmul(su.scale, u.im));
    }
  }
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < CW; ++q) acc += sum.get(q);
  acc *= sw.inv * (su.inv * su.inv);
  const double v = block_sum(acc, red);
  if (threadIdx.x == 0) part[SL_KIN * kPartStride + blockIdx.x] = v;
}

struct SlotCounts {
  int n[NSLOT];
};

__global__ void __launch_bounds__(256) k_sum_slots(const double* part, SlotCounts cnt, double* out) {
  __shared__ double red[32];
  const int s = blockIdx.x;
  double acc = 0.0;
  for (int i = threadIdx.x; i < cnt.n[s]; i += blockDim.x) acc += part[s * kPartStride + i];
  const double v = block_sum(acc, red);
  if (threadIdx.x == 0) out[s] = v;
}

// ---------------------------------------------------------------------------
// Optional float64 renormalisation of the float32 path (not part of the
// paper's scheme): hold the mass at its value at the start of each fse_step
// call. Pass E (or XI) writes per-tile partial masses, k_renorm turns them
// into sqrt(N0 / N), pass A multiplies u2 by it.
// ---------------------------------------------------------------------------
constexpr int kRenormSlot = 15;
constexpr long long kScalarBase = 16LL * kPartStride;

template <typename Real>
__global__ void __launch_bounds__(256) k_sumsq(const typename Cplx<Real>::T* __restrict__ psi, long long N,
                                               double* part) {
  __shared__ double red[32];
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const typename Cplx<Real>::T u = psi[i];
    acc += (double)u.x * u.x + (double)u.y * u.y;
  }
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

__global__ void __launch_bounds__(256) k_renorm(const double* part, int count, double* scal, int init) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += part[i];
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) {
    if (init) scal[0] = acc;
    else scal[1] = acc > 0.0 ? sqrt(scal[0] / acc) : 1.0;
  }
}

double* renorm_part(fse_plan* P) {
  return reinterpret_cast<double*>(P->ws_ptr(P->off_red)) + kRenormSlot * kPartStride;
}
const double* renorm_scale(fse_plan* P) {
  return reinterpret_cast<double*>(P->ws_ptr(P->off_red)) + kScalarBase + 1;
}

fse_status renorm_begin(fse_plan* P, const void* psi) {
  const long long N = (long long)P->nx * P->ny * P->nz;
  const int blocks = (int)std::min<long long>(kRedBlocks, (N + 255) / 256);
  double* scal = reinterpret_cast<double*>(P->ws_ptr(P->off_red)) + kScalarBase;
  cudaEvent_t ev = prof_begin(P);
  if (P->prec == FSE_F32)
    k_sumsq<float><<<blocks, 256, 0, P->stream>>>(reinterpret_cast<const float2*>(psi), N, renorm_part(P));
  else
    k_sumsq<double><<<blocks, 256, 0, P->stream>>>(reinterpret_cast<const double2*>(psi), N, renorm_part(P));
  prof_end(P, FSE_PASS_OTHER, ev);
  fse_status st = launched(P, cudaGetLastError(), "renormalisation");
  if (st != FSE_OK) return st;
  k_renorm<<<1, 256, 0, P->stream>>>(renorm_part(P), blocks, scal, 1);
  return launched(P, cudaGetLastError(), "renormalisation");
}

fse_status renorm_step(fse_plan* P, int count) {
  if (count > kPartStride) return fail(P, FSE_ERR_UNSUPPORTED, "renormalisation: grid too large");
  double* scal = reinterpret_cast<double*>(P->ws_ptr(P->off_red)) + kScalarBase;
  cudaEvent_t ev = prof_begin(P);
  k_renorm<<<1, 256, 0, P->stream>>>(renorm_part(P), count, scal, 0);
  prof_end(P, FSE_PASS_OTHER, ev);
  return launched(P, cudaGetLastError(), "renormalisation");
}

template <typename Real>
fse_status fft_full(fse_plan* P, void* buf, int dir) {
  MulArgs m;
  std::memset(&m, 0, sizeof(m));
  XArgs xa = x_args(P, buf, nullptr);
  fse_status st;
  ColArgs ay{buf, (long long)P->nx * P->ny, P->nx, P->nz, P->nx};
  ColArgs az{buf, P->nx, (long long)P->nx * P->ny, P->ny, P->nx};
  if (dir < 0) {
    if ((st = xpass(P, XP_FWD, xa)) != FSE_OK) return st;
    if ((st = col(P, FSE_PASS_OTHER, P->ny, COL_FWD, ay, m)) != FSE_OK) return st;
    if (P->dim == 3 && (st = col(P, FSE_PASS_OTHER, P->nz, COL_FWD, az, m)) != FSE_OK) return st;
    return FSE_OK;
  }
  if (P->dim == 3 && (st = col(P, FSE_PASS_OTHER, P->nz, COL_INV, az, m)) != FSE_OK) return st;
  if ((st = col(P, FSE_PASS_OTHER, P->ny, COL_INV, ay, m)) != FSE_OK) return st;
  return xpass(P, XP_INV, xa);
}

template fse_status fft_full<float>(fse_plan*, void*, int);
template fse_status fft_full<double>(fse_plan*, void*, int);

fse_status nonlocal_field(fse_plan* P, const void* psi, const double* mdir, void* phi) {
  void* spec = P->ws_ptr(P->off_spec);
  fse_status st;
  XArgs xa = x_args(P, const_cast<void*>(psi), spec);
  if ((st = xpass(P, XP_D, xa)) != FSE_OK) return st;  // S = R2C of rho
  const double* md = mdir ? mdir : P->p.dip_n;
  if ((st = nonlocal_yz(P, spec, 0.0, 0.0, false, md, 1.0)) != FSE_OK) return st;
  xa.out = phi;
  return xpass(P, XP_R, xa);
}

template <typename Real>
fse_status observables(fse_plan* P, const void* psi_in, double t, const double* gam, fse_obs* out) {
  typedef typename Cplx<Real>::T C;
  const C* psi = reinterpret_cast<const C*>(psi_in);
  C* tmp = reinterpret_cast<C*>(P->ws_ptr(P->off_tmp));
  C* spec = reinterpret_cast<C*>(P->ws_ptr(P->off_spec));
  double* part = reinterpret_cast<double*>(P->ws_ptr(P->off_red));
  double* sums = part + NSLOT * kPartStride;
  cudaError_t e;
  fse_status st;
  SlotCounts cnt;
  for (int k = 0; k < NSLOT; ++k) cnt.n[k] = 0;

  ObsArgs o;
  o.nx = P->nx;
  o.ny = P->ny;
  o.nlines = P->ny * P->nz;
  for (int j = 0; j < 3; ++j) {
    o.lo[j] = j < P->dim ? P->p.lo[j] : 0.0;
    o.h[j] = P->h[j];
    const double g = j < P->dim ? (gam ? gam[j] : P->p.gamma[j]) : 0.0;
    o.g2[j] = 0.5 * g * g;
    o.ic[j] = j < P->dim ? origin_index(P, j) : 0;
    o.lat_k[j] = j < P->dim ? P->p.lat_k[j] : 0.0;
  }
  o.c = std::cos(P->p.omega * t);
  o.s = std::sin(P->p.omega * t);
  // In a turned frame the moments give a trap's energy up to rounding of that of
  // its stiff axis in all directions: for a cloud along the soft axis of frequencies
  // 100 : 1 it was 6e-14 off, summed point by point 1e-16, as it is beyond 2 : 1
  // (observables of 128^3 float32 fields without interaction 130 -> 180 us).
  const double stiff = std::fmax(o.g2[0], o.g2[1]), soft = std::fmin(o.g2[0], o.g2[1]);
  o.by_points = o.s != 0.0 && !(stiff <= 4.0 * soft);
  o.lat_amp = P->p.lat_amp;
  const long long N = (long long)P->nx * P->ny * P->nz;
  const int blocks = std::min(2 * kSMs, (o.nlines + 7) / 8);

  // nonlocal energy density: Phi = U~(., t) * rho (un-integrated kernel at time t)
  if (has_nonlocal(P)) {
    XArgs xr = x_args(P, const_cast<C*>(psi), spec);
    if ((st = xpass(P, XP_D, xr)) != FSE_OK) return st;  // S = R2C of rho
    double mdir[3] = {0, 0, 0};
    if (P->p.kernel == FSE_KERNEL_DDI3D || P->p.kernel == FSE_KERNEL_DDI2D) {
      // m(t) = A(t)^T n
      const double n1 = P->p.dip_n[0], n2 = P->p.dip_n[1], n3 = P->p.dip_n[2];
      mdir[0] = o.c * n1 - o.s * n2;
      mdir[1] = o.s * n1 + o.c * n2;
      mdir[2] = n3;
    }
    if ((st = nonlocal_yz(P, spec, t, t, false, mdir, 1.0)) != FSE_OK) return st;
    xr.part = part + SL_NON * kPartStride;
    if (x_tiles(P, xr.nlines) > kPartStride) return fail(P, FSE_ERR_UNSUPPORTED, "observables: grid too large");
    if ((st = xpass(P, XP_R, xr)) != FSE_OK) return st;
    cnt.n[SL_NON] = x_tiles(P, xr.nlines);
  }

  cudaEvent_t ev = prof_begin(P);
  k_obs_phys<<<blocks, 256, 0, P->stream>>>(psi, o, part);
  prof_end(P, FSE_PASS_OTHER, ev);
  if ((st = launched(P, cudaGetLastError(), "observables")) != FSE_OK) return st;
  for (int k = SL_MASS; k <= SL_XY; ++k) cnt.n[k] = blocks;

  // spectrum of psi (in the scratch field)
  const double dkx = 2 * kPi / (P->p.hi[0] - P->p.lo[0]);
  const double dky = 2 * kPi / (P->p.hi[1] - P->p.lo[1]);
  const double dkz = P->dim == 3 ? 2 * kPi / (P->p.hi[2] - P->p.lo[2]) : 0.0;
  MulArgs m;
  std::memset(&m, 0, sizeof(m));
  XArgs x0 = x_args(P, tmp, nullptr);
  x0.aux = psi;
  if ((st = xpass(P, XP_FWD, x0)) != FSE_OK) return st;
  ColArgs ay{tmp, (long long)P->nx * P->ny, P->nx, P->nz, P->nx};
  if ((st = col(P, FSE_PASS_OTHER, P->ny, COL_FWD, ay, m)) != FSE_OK) return st;
  if (P->dim == 3) {
    ColArgs az{tmp, P->nx, (long long)P->nx * P->ny, P->ny, P->nx};
    if ((st = col(P, FSE_PASS_OTHER, P->nz, COL_FWD, az, m)) != FSE_OK) return st;
  }
  ev = prof_begin(P);
  k_obs_kin<Real><<<blocks, 256, 0, P->stream>>>(tmp, o, P->nz, dkx, dky, dkz, P->p.s, P->p.m * P->p.m, part);
  prof_end(P, FSE_PASS_OTHER, ev);
  if ((st = launched(P, cudaGetLastError(), "observables")) != FSE_OK) return st;
  cnt.n[SL_KIN] = blocks;

  // <L_z> = Im sum conj(psi) (x d_y - y d_x) psi: each derivative needs the
  // transforms of its own axis alone, and its product with psi is summed where
  // it is formed
  XArgs xl = x_args(P, const_cast<C*>(psi), nullptr);
  xl.beta_dt = dkx / P->nx;
  xl.part = part + SL_LZX * kPartStride;
  if (x_tiles(P, xl.nlines) > kPartStride) return fail(P, FSE_ERR_UNSUPPORTED, "observables: grid too large");
  if ((st = xpass(P, XP_LZ, xl)) != FSE_OK) return st;
  cnt.n[SL_LZX] = x_tiles(P, xl.nlines);
  m.dkr = dky / P->ny;
  ColArgs al{const_cast<C*>(psi), (long long)P->nx * P->ny, P->nx, P->nz, P->nx};
  al.part = part + SL_LZY * kPartStride;
  al.lo = o.lo[0];
  al.h = o.h[0];
  int lz_blocks = 0;
  al.blocks_out = &lz_blocks;
  if ((st = col(P, FSE_PASS_OTHER, P->ny, COL_LZ, al, m)) != FSE_OK) return st;
  cnt.n[SL_LZY] = lz_blocks;

  k_sum_slots<<<NSLOT, 256, 0, P->stream>>>(part, cnt, sums);
  if ((st = launched(P, cudaGetLastError(), "observables")) != FSE_OK) return st;
  double h[NSLOT];
  if ((e = cudaMemcpyAsync(h, sums, sizeof(h), cudaMemcpyDeviceToHost, P->stream)) != cudaSuccess)
    return cuda_fail(P, e, "observables read");
  if ((e = cudaStreamSynchronize(P->stream)) != cudaSuccess) return cuda_fail(P, e, "observables sync");

  double hd = 1.0;
  for (int j = 0; j < P->dim; ++j) hd *= P->h[j];
  // sums in index units -> coordinates x = c + h i
  {
    double c[3];
    for (int j = 0; j < 3; ++j) c[j] = j < P->dim ? o.lo[j] + o.h[j] * o.ic[j] : 0.0;
    const double s0 = h[SL_MASS], i1[3] = {h[SL_X], h[SL_Y], h[SL_Z]};
    h[SL_XY] = c[0] * c[1] * s0 + c[0] * o.h[1] * i1[1] + c[1] * o.h[0] * i1[0] + o.h[0] * o.h[1] * h[SL_XY];
    for (int j = 0; j < 3; ++j) {
      h[SL_XX + j] = c[j] * c[j] * s0 + 2 * c[j] * o.h[j] * i1[j] + o.h[j] * o.h[j] * h[SL_XX + j];
      h[SL_X + j] = c[j] * s0 + o.h[j] * i1[j];
    }
  }
  std::memset(out, 0, sizeof(*out));
  out->mass = hd * h[SL_MASS];
  out->e_kin = 0.5 * hd / (double)N * h[SL_KIN];
  // W = g2_x X^2 + g2_y Y^2 + g2_z z^2 (+ lattice), X = c x + s y, Y = -s x + c y
  double trap = o.g2[2] * h[SL_ZZ];
  if (!o.by_points)
    trap += o.g2[0] * (o.c * o.c * h[SL_XX] + 2 * o.c * o.s * h[SL_XY] + o.s * o.s * h[SL_YY]) +
            o.g2[1] * (o.s * o.s * h[SL_XX] - 2 * o.c * o.s * h[SL_XY] + o.c * o.c * h[SL_YY]);
  out->e_pot = hd * (h[SL_WRHO] + trap);
  out->e_int = 0.5 * P->p.beta * hd * h[SL_RHO2];
  out->e_non = has_nonlocal(P) ? 0.5 * P->p.lambda * hd * h[SL_NON] : 0.0;
  out->lz = hd * (h[SL_LZY] + h[SL_LZX]);
  out->e_rot = -P->p.omega * out->lz;
  out->energy = out->e_kin + out->e_pot + out->e_int + out->e_non + out->e_rot;
  const double xt[3] = {hd * h[SL_X], hd * h[SL_Y], hd * h[SL_Z]};
  out->xc[0] = o.c * xt[0] + o.s * xt[1];
  out->xc[1] = -o.s * xt[0] + o.c * xt[1];
  out->xc[2] = P->dim == 3 ? xt[2] : 0.0;
  const double Sxx = hd * h[SL_XX], Syy = hd * h[SL_YY], Sxy = hd * h[SL_XY];
  out->width[0] = o.c * o.c * Sxx + 2 * o.c * o.s * Sxy + o.s * o.s * Syy;
  out->width[1] = o.s * o.s * Sxx - 2 * o.c * o.s * Sxy + o.c * o.c * Syy;
  out->width[2] = P->dim == 3 ? hd * h[SL_ZZ] : 0.0;
  if (!std::isfinite(out->mass) || !std::isfinite(out->energy))
    return fail(P, FSE_ERR_NONFINITE, "observables: non-finite mass or energy");
  return FSE_OK;
}

}  // namespace fse

using namespace fse;

extern "C" fse_status fse_observables(fse_plan_t P, const void* psi, double t, const double* gamma, fse_obs* out) {
  if (!P || !psi || !out) return FSE_ERR_INVALID;
  if (!P->ws || !P->precomputed) return fail(P, FSE_ERR_INVALID, "fse_kernel_precompute has not run");
  return P->prec == FSE_F32 ? observables<float>(P, psi, t, gamma, out) : observables<double>(P, psi, t, gamma, out);
}
