// fse_ground.cu -- ground state by GF-GauSum (Section 3.2, Eqs. gf-eq2, gf-colb2, gffg33),
// and the shifted and kicked initial data of the dynamics runs (Section 4.3, Eq. ini_dyn).
//
// Gradient flow with discrete normalisation, discretised by backward Euler:
//   (1/dt + (-Lap + m^2)^s / 2 + W_n - Omega L_z) phi^(1) = phi^n / dt,
//   W_n = V + beta |phi^n|^2 + lambda Phi^n,  Phi^n = U * |phi^n|^2,
//   phi^{n+1} = phi^(1) / ||phi^(1)||,
// each step solved by BiCGStab on the left system of Eq. precond_type1,
//   (I + P_Delta A_TF) phi^(1) = P_Delta phi^n / dt,
//   P_Delta = [1/dt + (|k|^2 + m^2)^s / 2]^-1,  A_TF = W_n - Omega L_z,
// with L_z = -i (x d_y - y d_x) by spectral derivatives. The problem is posed
// in the laboratory frame: V is the trap (harmonic plus optional lattice) and
// the dipole axis is n. Every transform runs through the plan's FFT passes;
// the BiCGStab vectors live in a caller-supplied workspace, and its scalars
// (inner products, alpha, omega, beta, the residual) stay on the device: the
// host reads them one iteration behind the GPU to stop the solve.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "fse.h"
#include "fse_internal.h"
#include "fse_gsx.cuh"

namespace fse {
namespace {

constexpr int kGsBlocks = 1024;  // blocks of the elementwise kernels, at most

struct GsGrid {
  int nx, ny, nz;
  double lo[3], h[3], dk[3];
};

__device__ __forceinline__ void gs_index(long long i, const GsGrid& g, int& ix, int& iy, int& iz) {
  ix = (int)(i % g.nx);
  const long long r = i / g.nx;
  iy = (int)(r % g.ny);
  iz = (int)(r / g.ny);
}

// P_Delta / N on the octant |p_j| = 0..n_j/2 of the spectrum: 1 / (N (1/dt + (|k|^2 + m^2)^s / 2))
template <typename Real>
__global__ void k_gs_precond_table(Real* pk, GsGrid g, double inv_dt, double s, double m2, double inv_n) {
  const int hx = g.nx / 2 + 1, hy = g.ny / 2 + 1, hz = g.nz > 1 ? g.nz / 2 + 1 : 1;
  const long long N = (long long)hx * hy * hz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const int ix = (int)(i % hx);
    const long long r = i / hx;
    const double kx = g.dk[0] * ix, ky = g.dk[1] * (int)(r % hy), kz = g.dk[2] * (int)(r / hy);
    const double k2 = kx * kx + ky * ky + kz * kz + m2;
    pk[i] = Real(inv_n / (inv_dt + 0.5 * (k2 > 0.0 ? pow(k2, s) : 0.0)));
  }
}

// W = V + beta |phi|^2 + lambda Phi, V = sum_v gamma_v^2 x_v^2 / 2 + lat_amp sum_v sin^2(lat_k_v x_v)
template <typename Real>
__global__ void k_gs_potential(const typename Cplx<Real>::T* __restrict__ phi, const Real* __restrict__ Phi,
                               Real* __restrict__ W, GsGrid g, double3 g2, double beta, double lam, double lat_amp,
                               double3 lk) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz;
    gs_index(i, g, ix, iy, iz);
    const double x = g.lo[0] + g.h[0] * ix, y = g.lo[1] + g.h[1] * iy, z = g.lo[2] + g.h[2] * iz;
    double v = g2.x * x * x + g2.y * y * y + g2.z * z * z;
    if (lat_amp != 0.0) {
      const double sx = sin(lk.x * x), sy = sin(lk.y * y), sz = sin(lk.z * z);
      v += lat_amp * (sx * sx + sy * sy + sz * sz);
    }
    const typename Cplx<Real>::T u = phi[i];
    v += beta * ((double)u.x * u.x + (double)u.y * u.y);
    if (Phi) v += lam * (double)Phi[i];
    W[i] = Real(v);
  }
}

// Partials of sum |a|^2 (float64), part[block]
template <typename Real>
__global__ void __launch_bounds__(256) k_gs_norm(const typename Cplx<Real>::T* a, long long N, double* part) {
  __shared__ double red[32];
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const typename Cplx<Real>::T x = a[i];
    acc += (double)x.x * x.x + (double)x.y * x.y;
  }
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// x <- x / ||x|| with ||x||^2 = hd * norm[0], and (old non-null) partials of max |x - old|.
// A norm that is not positive (the host then returns an error) leaves x as it is.
template <typename Real>
__global__ void __launch_bounds__(256) k_gs_normalise(typename Cplx<Real>::T* x, const typename Cplx<Real>::T* old,
                                                      const double* norm, double hd, long long N, double* part) {
  __shared__ double red[256];
  if (!(norm[0] > 0.0)) return;
  const Real f = Real(1.0 / sqrt(hd * norm[0]));
  double m = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    typename Cplx<Real>::T u = x[i];
    u = mk(u.x * f, u.y * f);
    x[i] = u;
    if (old) {
      const double dx = (double)u.x - old[i].x, dy = (double)u.y - old[i].y;
      m = fmax(m, dx * dx + dy * dy);
      if (!(dx * dx + dy * dy >= 0.0)) m = __longlong_as_double(0x7ff0000000000000LL);  // NaN shows as infinity
    }
  }
  if (!old) return;
  red[threadIdx.x] = m;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sqrt(red[0]);
}

// ---------------------------------------------------------------------------
// BiCGStab scalars on the device. The state sc[] holds, in float64,
//   rho (complex, sc[0..1]), rho_prev (sc[2..3]), alpha (sc[4..5]),
//   omega (sc[6..7]), beta (sc[8..9]), ||b|| (sc[10]), ||r|| / ||b|| (sc[11]),
//   done (sc[12]: converged or broken down), iterations (sc[13]), tol (sc[14]).
// One block sums the partials of an inner product in a fixed order and its
// first thread updates the state; the vector updates read their coefficients
// from it, so an inner iteration needs no host round trip. Once done is set,
// every update leaves its output untouched.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 zdiv(double2 a, double2 b) {
  const double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ void st2(double* p, double2 v) {
  p[0] = v.x;
  p[1] = v.y;
}

// after <b, b>, <r, r> (r = b - M x, rh = r): the start of an inner solve
__device__ __forceinline__ void gs_sc_init(double* sc, const double* out, double tol) {
  const double bn = sqrt(out[0]);
  const double res = bn > 0.0 ? sqrt(out[2]) / bn : 0.0;
  st2(sc + SC_RHO, make_double2(out[2], 0.0));
  st2(sc + SC_RHOP, make_double2(1.0, 0.0));
  st2(sc + SC_ALPHA, make_double2(1.0, 0.0));
  st2(sc + SC_OM, make_double2(1.0, 0.0));
  st2(sc + SC_BETA, make_double2(0.0, 0.0));
  sc[SC_BN] = bn;
  sc[SC_RES] = res;
  sc[SC_TOL] = tol;
  sc[SC_IT] = 0.0;
  sc[SC_DONE] = (!(res > tol) || out[2] == 0.0) ? 1.0 : 0.0;
}

// after <rh, v>: alpha = rho / <rh, v> (breakdown when it vanishes)
__device__ __forceinline__ void gs_sc_alpha(double* sc, const double* out) {
  if (sc[SC_DONE] != 0.0) return;
  const double2 rv = make_double2(out[0], out[1]);
  if (rv.x == 0.0 && rv.y == 0.0) {
    sc[SC_DONE] = 1.0;
    return;
  }
  st2(sc + SC_ALPHA, zdiv(gs_ld2(sc + SC_RHO), rv));
}

// after <t, s>, <t, t>: omega = <t, s> / <t, t> (0 if <t, t> = 0)
__device__ __forceinline__ void gs_sc_omega(double* sc, const double* out) {
  if (sc[SC_DONE] != 0.0) return;
  st2(sc + SC_OM, out[2] > 0.0 ? make_double2(out[0] / out[2], out[1] / out[2]) : make_double2(0.0, 0.0));
}

// after <rh, r>, <r, r>: the end of an iteration
__device__ __forceinline__ void gs_sc_rho(double* sc, const double* out) {
  if (sc[SC_DONE] != 0.0) return;
  const double2 rho_prev = gs_ld2(sc + SC_RHO), rho = make_double2(out[0], out[1]);
  const double2 alpha = gs_ld2(sc + SC_ALPHA), om = gs_ld2(sc + SC_OM);
  st2(sc + SC_RHOP, rho_prev);
  st2(sc + SC_RHO, rho);
  const double res = sqrt(out[2]) / sc[SC_BN];
  sc[SC_RES] = res;
  sc[SC_IT] += 1.0;
  const bool om0 = om.x == 0.0 && om.y == 0.0, rho0 = rho.x == 0.0 && rho.y == 0.0;
  if (om0 || rho0 || !(res > sc[SC_TOL])) {
    sc[SC_DONE] = 1.0;
    return;
  }
  // beta of the next iteration: (rho / rho_prev) (alpha / omega)
  st2(sc + SC_BETA, gs_mul(zdiv(rho, rho_prev), zdiv(alpha, om)));
}

enum { FIN_SUM = 0, FIN_MAX = 1, FIN_INIT = 2, FIN_ALPHA = 3, FIN_OMEGA = 4, FIN_RHO = 5 };
// out[v] = sum (FIN_MAX: max) of the count partials of value v, v < nv <= 4 (64
// threads each, fixed order), then the scalar update that waits for them
template <int MODE>
__global__ void __launch_bounds__(256) k_gs_fin(const double* part, int stride, int count, int nv, double* out, double* sc,
                                                double tol) {
  pass_prologue();
  __shared__ double red[256];
  const int v = threadIdx.x >> 6, t = threadIdx.x & 63;
  double acc = 0.0;
  if (v < nv)
    for (int i = t; i < count; i += 64) {
      const double x = part[(long long)v * stride + i];
      acc = MODE == FIN_MAX ? fmax(acc, x) : acc + x;
    }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 32; o > 0; o >>= 1) {
    if (t < o) red[threadIdx.x] = MODE == FIN_MAX ? fmax(acc, red[threadIdx.x + o]) : acc + red[threadIdx.x + o];
    __syncthreads();
    acc = red[threadIdx.x];
  }
  if (t == 0 && v < nv) out[v] = acc;
  if (threadIdx.x != 0) return;
  const double o4[4] = {red[0], red[64], red[128], red[192]};
  if (MODE == FIN_INIT) gs_sc_init(sc, o4, tol);
  if (MODE == FIN_ALPHA) gs_sc_alpha(sc, o4);
  if (MODE == FIN_OMEGA) gs_sc_omega(sc, o4);
  if (MODE == FIN_RHO) gs_sc_rho(sc, o4);
}

// The end of an iteration: x += alpha p + omega s, r = s - omega t (nothing
// when done), and the partials of <rh, r>, <r, r>.
template <typename Real>
__global__ void __launch_bounds__(256) k_gs_update(typename Cplx<Real>::T* x, typename Cplx<Real>::T* r,
                                                   const typename Cplx<Real>::T* p, const typename Cplx<Real>::T* s,
                                                   const typename Cplx<Real>::T* t, const typename Cplx<Real>::T* rh,
                                                   const double* sc, long long N, double* part, int stride) {
  typedef typename Cplx<Real>::T C;
  pass_prologue();
  __shared__ double red[3 * 256];
  double acc[3] = {0, 0, 0};
  const bool done = sc[SC_DONE] != 0.0;
  const double2 al = gs_ld2(sc + SC_ALPHA), om = gs_ld2(sc + SC_OM);
  const C a = mk(Real(al.x), Real(al.y)), w = mk(Real(om.x), Real(om.y));
  if (!done)
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
      const C si = s[i], pi = p[i], ti = t[i], hi = rh[i];
      C xi = x[i];
      xi = mk(xi.x + a.x * pi.x - a.y * pi.y + w.x * si.x - w.y * si.y, xi.y + a.x * pi.y + a.y * pi.x + w.x * si.y + w.y * si.x);
      const C ri = mk(si.x - w.x * ti.x + w.y * ti.y, si.y - w.x * ti.y - w.y * ti.x);
      x[i] = xi;
      r[i] = ri;
      acc[0] += (double)hi.x * ri.x + (double)hi.y * ri.y;
      acc[1] += (double)hi.x * ri.y - (double)hi.y * ri.x;
      acc[2] += (double)ri.x * ri.x + (double)ri.y * ri.y;
    }
  block_sums(acc, red, [&](int v, double z) { part[(long long)v * stride + blockIdx.x] = z; });
}

// Spectral translation by x0 (the Nyquist mode takes cos(k_N x0), the mean of
// its two aliases) and 1/N for the unnormalised inverse.
template <typename Real>
__global__ void k_gs_shift(typename Cplx<Real>::T* __restrict__ sp, GsGrid g, double3 x0, double inv_n) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz;
    gs_index(i, g, ix, iy, iz);
    const int nn[3] = {g.nx, g.ny, g.nz};
    const int id[3] = {ix, iy, iz};
    const double xs[3] = {x0.x, x0.y, x0.z};
    double re = inv_n, im = 0.0;
    for (int j = 0; j < 3; ++j) {
      if (nn[j] == 1 || xs[j] == 0.0) continue;
      const double k = g.dk[j] * wrap_index(id[j], nn[j]);
      double c, s;
      if (2 * id[j] == nn[j]) {
        c = cos(k * xs[j]);
        s = 0.0;
      } else {
        sincos(-k * xs[j], &s, &c);
      }
      const double r2 = re * c - im * s, i2 = re * s + im * c;
      re = r2;
      im = i2;
    }
    const typename Cplx<Real>::T u = sp[i];
    sp[i] = mk(Real(re * u.x - im * u.y), Real(re * u.y + im * u.x));
  }
}

// psi *= exp(i k . x)
template <typename Real>
__global__ void k_gs_kick(typename Cplx<Real>::T* __restrict__ psi, GsGrid g, double3 kv) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz;
    gs_index(i, g, ix, iy, iz);
    const double ph = kv.x * (g.lo[0] + g.h[0] * ix) + kv.y * (g.lo[1] + g.h[1] * iy) + kv.z * (g.lo[2] + g.h[2] * iz);
    double s, c;
    sincos(ph, &s, &c);
    const typename Cplx<Real>::T u = psi[i];
    psi[i] = mk(Real(c * u.x - s * u.y), Real(c * u.y + s * u.x));
  }
}

GsGrid gs_grid(const fse_plan* P) {
  GsGrid g;
  g.nx = P->nx;
  g.ny = P->ny;
  g.nz = P->nz;
  for (int j = 0; j < 3; ++j) {
    g.lo[j] = j < P->dim ? P->p.lo[j] : 0.0;
    g.h[j] = j < P->dim ? P->h[j] : 0.0;
    g.dk[j] = j < P->dim ? 2 * kPi / (P->p.hi[j] - P->p.lo[j]) : 0.0;
  }
  return g;
}

template <typename Real>
fse_status shift_kick(fse_plan* P, void* psi, const double* x0, const double* kv) {
  const GsGrid g = gs_grid(P);
  const long long N = (long long)P->nx * P->ny * P->nz;
  const int blocks = (int)std::min<long long>(kGsBlocks, (N + 255) / 256);
  fse_status st;
  if (x0 && (x0[0] != 0.0 || x0[1] != 0.0 || (P->dim == 3 && x0[2] != 0.0))) {
    if ((st = fft_full<Real>(P, psi, -1)) != FSE_OK) return st;
    k_gs_shift<Real><<<blocks, 256, 0, P->stream>>>(static_cast<typename Cplx<Real>::T*>(psi), g,
                                                    make_double3(x0[0], x0[1], P->dim == 3 ? x0[2] : 0.0),
                                                    1.0 / (double)N);
    if ((st = launched(P, cudaGetLastError(), "shift")) != FSE_OK) return st;
    if ((st = fft_full<Real>(P, psi, +1)) != FSE_OK) return st;
  }
  if (kv && (kv[0] != 0.0 || kv[1] != 0.0 || (P->dim == 3 && kv[2] != 0.0))) {
    k_gs_kick<Real><<<blocks, 256, 0, P->stream>>>(static_cast<typename Cplx<Real>::T*>(psi), g,
                                                   make_double3(kv[0], kv[1], P->dim == 3 ? kv[2] : 0.0));
    if ((st = launched(P, cudaGetLastError(), "kick")) != FSE_OK) return st;
  }
  return FSE_OK;
}

size_t al256(size_t v) { return (v + 255) & ~(size_t)255; }

// partials per value: one per tile of the x passes or block of the vector kernels
int gs_parts(const fse_plan* P) {
  const int t = x_tiles(const_cast<fse_plan*>(P), P->ny * (P->dim == 3 ? P->nz : 1));
  return t > kGsBlocks ? t : kGsBlocks;
}

// workspace: 8 complex fields (the last one only used with rotation), 3 real
// fields, reduction partials and results
struct GsLayout {
  size_t cplx[8], real[3], part, out, sc, total;
};
GsLayout gs_layout(const fse_plan* P) {
  GsLayout L;
  const size_t N = (size_t)P->nx * P->ny * P->nz;
  size_t off = 0;
  for (int i = 0; i < 8; ++i) {
    L.cplx[i] = off;
    off = al256(off + N * P->csize);
  }
  for (int i = 0; i < 3; ++i) {
    L.real[i] = off;
    off = al256(off + N * P->rsize);
  }
  L.part = off;
  off = al256(off + sizeof(double) * 4 * gs_parts(P));
  L.out = off;
  off = al256(off + sizeof(double) * 8);
  L.sc = off;
  off = al256(off + sizeof(double) * SC_SIZE);
  L.total = off;
  return L;
}

template <typename Real>
struct Gs {
  typedef typename Cplx<Real>::T C;
  fse_plan* P;
  cudaStream_t st;
  long long N;
  int blocks, nlines, tiles, stride;
  GsGrid g;
  C *phin, *r, *rh, *p, *v, *s, *t, *w;  // w: the operator's work field
  C* dy;
  Real *W, *pk, *Phi;
  double *part, *out, *sc;
  double omega;

  fse_status chk(const char* w0) { return launched(P, cudaGetLastError(), w0); }
  fse_status copy(C* dst, const C* src) {
    cudaError_t e = cudaMemcpyAsync(dst, src, (size_t)N * sizeof(C), cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? FSE_OK : cuda_fail(P, e, "ground state copy");
  }
  template <int MODE> fse_status fin(int count, int nv, double tol = 0.0) {
    return launched(P, launch_pass(k_gs_fin<MODE>, 1, 256, 0, st, (const double*)part, stride, count, nv, out, sc, tol),
                    "ground state reduction");
  }
  // the passes along y (and z) of P_Delta on the x-spectrum in w
  fse_status precond_yz() {
    MulArgs m;
    std::memset(&m, 0, sizeof(m));
    m.kin = pk;
    m.lx = P->nx;
    ColArgs ay{w, (long long)P->nx * P->ny, P->nx, P->nz, P->nx};
    if (P->dim == 2) {
      m.kin_sr = P->nx / 2 + 1;
      return col(P, FSE_PASS_OTHER, P->ny, COL_RMUL, ay, m);
    }
    fse_status s0;
    if ((s0 = col(P, FSE_PASS_OTHER, P->ny, COL_FWD, ay, m)) != FSE_OK) return s0;
    m.lp = P->ny;
    m.kin_sp = P->nx / 2 + 1;
    m.kin_sr = (long long)(P->nx / 2 + 1) * (P->ny / 2 + 1);
    ColArgs az{w, P->nx, (long long)P->nx * P->ny, P->ny, P->nx};
    if ((s0 = col(P, FSE_PASS_OTHER, P->nz, COL_RMUL, az, m)) != FSE_OK) return s0;
    return col(P, FSE_PASS_OTHER, P->ny, COL_INV, ay, m);
  }
  // d_y of u into dy (rotation)
  fse_status deriv_y(const C* u) {
    MulArgs m;
    std::memset(&m, 0, sizeof(m));
    m.dkr = g.dk[1] / P->ny;
    ColArgs a{const_cast<C*>(u), (long long)P->nx * P->ny, P->nx, P->nz, P->nx};
    a.out = dy;
    return col(P, FSE_PASS_OTHER, P->ny, COL_DY, a, m);
  }
  // w = x-spectrum of A_TF u (or scale u), u by `mode` from a, c, o; with
  // rotation u itself has to exist before its derivative along y is taken
  fse_status fwd(int mode, const C* a, const C* c, C* o, const Real* Wf, double scale) {
    GsFwd f;
    std::memset(&f, 0, sizeof(f));
    f.mode = mode;
    f.nlines = nlines;
    f.ny = P->ny;
    f.a = a;
    f.c = c;
    f.o = o;
    f.W = Wf;
    f.scale = scale;
    f.omega = omega;
    f.lo0 = g.lo[0];
    f.h0 = g.h[0];
    f.lo1 = g.lo[1];
    f.h1 = g.h[1];
    f.dkx = g.dk[0];
    f.sc = sc;
    f.out = w;
    fse_status s0;
    if (omega != 0.0 && Wf) {
      const C* u = a;
      if (mode != U_PLAIN) {
        // u into o (its x-spectrum, also computed, is overwritten below)
        f.W = nullptr;
        if ((s0 = launched(P, launch_gs_fwd<Real>(P->nx, f, twiddle(P, P->nx), st), "ground state update")) != FSE_OK)
          return s0;
        u = o;
        f.mode = U_PLAIN;
        f.a = o;
        f.W = Wf;
      }
      if ((s0 = deriv_y(u)) != FSE_OK) return s0;
      f.dy = dy;
    }
    return launched(P, launch_gs_fwd<Real>(P->nx, f, twiddle(P, P->nx), st), "ground state operator");
  }
  fse_status inv(int mode, const C* u, const C* q, C* y, C* y2) {
    GsInv f;
    f.mode = mode;
    f.nlines = nlines;
    f.in = w;
    f.u = u;
    f.q = q;
    f.y = y;
    f.y2 = y2;
    f.part = part;
    f.stride = stride;
    return launched(P, launch_gs_inv<Real>(P->nx, f, twiddle(P, P->nx), st), "ground state operator");
  }
  // ||x||^2 / hd into out[0]
  fse_status norm(const C* x) {
    k_gs_norm<Real><<<blocks, 256, 0, st>>>(x, N, part);
    fse_status s0 = chk("ground state reduction");
    return s0 != FSE_OK ? s0 : fin<FIN_SUM>(blocks, 1);
  }
  // x <- x / ||x|| (norm in out[0]); with old also max |x - old| into out[1]
  fse_status normalise(C* x, const C* old, double hd) {
    k_gs_normalise<Real><<<blocks, 256, 0, st>>>(x, old, out, hd, N, part);
    fse_status s0 = chk("ground state normalisation");
    if (s0 != FSE_OK || !old) return s0;
    return launched(P, launch_pass(k_gs_fin<FIN_MAX>, 1, 256, 0, st, (const double*)part, stride, blocks, 1, out + 1, sc, 0.0),
                    "ground state reduction");
  }
  fse_status read(double* h, const double* d, int n) {
    cudaError_t e = cudaMemcpyAsync(h, d, sizeof(double) * n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? FSE_OK : cuda_fail(P, e, "ground state read");
  }
};

template <typename Real>
fse_status ground_state(fse_plan* P, void* psi_v, void* ws, const fse_gs_opts& o, fse_gs_info* info) {
  typedef typename Cplx<Real>::T C;
  const GsLayout L = gs_layout(P);
  char* base = static_cast<char*>(ws);
  Gs<Real> G;
  G.P = P;
  G.st = P->stream;
  G.N = (long long)P->nx * P->ny * P->nz;
  G.blocks = (int)std::min<long long>(2 * kSMs, (G.N + 255) / 256);
  G.nlines = P->ny * (P->dim == 3 ? P->nz : 1);
  G.tiles = x_tiles(P, G.nlines);
  G.stride = gs_parts(P);
  G.g = gs_grid(P);
  C** cp[8] = {&G.phin, &G.r, &G.rh, &G.p, &G.v, &G.s, &G.t, &G.dy};
  for (int i = 0; i < 8; ++i) *cp[i] = reinterpret_cast<C*>(base + L.cplx[i]);
  G.w = static_cast<C*>(P->ws_ptr(P->off_tmp));  // the plan's scratch field
  G.W = reinterpret_cast<Real*>(base + L.real[0]);
  G.pk = reinterpret_cast<Real*>(base + L.real[1]);
  G.Phi = reinterpret_cast<Real*>(base + L.real[2]);
  G.part = reinterpret_cast<double*>(base + L.part);
  G.out = reinterpret_cast<double*>(base + L.out);
  G.sc = reinterpret_cast<double*>(base + L.sc);
  G.omega = P->p.omega;
  C* x = static_cast<C*>(psi_v);
  const double hd = P->h[0] * P->h[1] * (P->dim == 3 ? P->h[2] : 1.0);
  const bool nl = has_nonlocal(P);
  fse_status st;
  double h2[2];

  k_gs_precond_table<Real><<<G.blocks, 256, 0, G.st>>>(G.pk, G.g, 1.0 / o.dt, P->p.s, P->p.m * P->p.m,
                                                       1.0 / (double)G.N);
  if ((st = G.chk("ground state preconditioner")) != FSE_OK) return st;
  if ((st = G.norm(x)) != FSE_OK || (st = G.read(h2, G.out, 1)) != FSE_OK) return st;
  if (!(h2[0] > 0.0)) return fail(P, FSE_ERR_INVALID, "ground state: zero initial field");
  if ((st = G.normalise(x, nullptr, hd)) != FSE_OK) return st;

  const double3 g2 = make_double3(0.5 * P->p.gamma[0] * P->p.gamma[0], 0.5 * P->p.gamma[1] * P->p.gamma[1],
                                  P->dim == 3 ? 0.5 * P->p.gamma[2] * P->p.gamma[2] : 0.0);
  const double3 lk = make_double3(P->p.lat_k[0], P->p.lat_k[1], P->dim == 3 ? P->p.lat_k[2] : 0.0);
  // one BiCGStab iteration: every operand and coefficient is on the device
  auto iteration = [&]() -> fse_status {
    fse_status s0;
    if ((s0 = G.fwd(U_P, G.r, G.v, G.p, G.W, 0.0)) != FSE_OK || (s0 = G.precond_yz()) != FSE_OK ||
        (s0 = G.inv(V_ADD, G.p, G.rh, G.v, nullptr)) != FSE_OK || (s0 = G.template fin<FIN_ALPHA>(G.tiles, 2)) != FSE_OK)
      return s0;
    if ((s0 = G.fwd(U_S, G.r, G.v, G.s, G.W, 0.0)) != FSE_OK || (s0 = G.precond_yz()) != FSE_OK ||
        (s0 = G.inv(V_ADD2, G.s, nullptr, G.t, nullptr)) != FSE_OK ||
        (s0 = G.template fin<FIN_OMEGA>(G.tiles, 3)) != FSE_OK)
      return s0;
    s0 = launched(P, launch_pass(k_gs_update<Real>, G.blocks, 256, 0, G.st, x, G.r, (const C*)G.p, (const C*)G.s,
                                 (const C*)G.t, (const C*)G.rh, (const double*)G.sc, G.N, G.part, G.stride),
                  "ground state update");
    return s0 != FSE_OK ? s0 : G.template fin<FIN_RHO>(G.blocks, 3);
  };
  int outer = 0;
  long long inner = 0;
  double change = 0.0, res = 0.0;
  while (outer < o.max_outer) {
    if ((st = G.copy(G.phin, x)) != FSE_OK) return st;
    if (nl && (st = nonlocal_field(P, x, nullptr, G.Phi)) != FSE_OK) return st;
    k_gs_potential<Real><<<G.blocks, 256, 0, G.st>>>(x, nl ? G.Phi : nullptr, G.W, G.g, g2, P->p.beta, P->p.lambda,
                                                      P->p.lat_amp, lk);
    if ((st = G.chk("ground state potential")) != FSE_OK) return st;
    // b = P_Delta phi^n / dt (held in s), r = b - M x, rh = r
    if ((st = G.fwd(U_PLAIN, x, nullptr, nullptr, nullptr, 1.0 / o.dt)) != FSE_OK || (st = G.precond_yz()) != FSE_OK ||
        (st = G.inv(V_SET, nullptr, nullptr, G.s, nullptr)) != FSE_OK)
      return st;
    if ((st = G.fwd(U_PLAIN, x, nullptr, nullptr, G.W, 0.0)) != FSE_OK || (st = G.precond_yz()) != FSE_OK ||
        (st = G.inv(V_RES, x, G.s, G.r, G.rh)) != FSE_OK ||
        (st = G.template fin<FIN_INIT>(G.tiles, 3, o.inner_tol)) != FSE_OK)
      return st;
    // Iterations are queued one ahead of the host: after queueing iteration
    // it, the host waits for the scalars of iteration it - 1 (copied to pinned
    // host memory behind it) and stops once they say done, so the GPU never
    // idles on a read-back; the extra iteration then changes nothing.
    double* hs = P->gs_host;
    int it = 0;
    for (; it < o.max_inner; ++it) {
      if ((st = iteration()) != FSE_OK) return st;
      cudaError_t e = cudaMemcpyAsync(hs + (it & 1) * SC_SIZE, G.sc, sizeof(double) * SC_SIZE,
                                      cudaMemcpyDeviceToHost, G.st);
      if (e == cudaSuccess) e = cudaEventRecord(P->gs_ev[it & 1], G.st);
      if (e != cudaSuccess) return cuda_fail(P, e, "ground state scalars");
      if (it >= 1) {
        if ((e = cudaEventSynchronize(P->gs_ev[(it - 1) & 1])) != cudaSuccess)
          return cuda_fail(P, e, "ground state scalars");
        if (hs[((it - 1) & 1) * SC_SIZE + SC_DONE] != 0.0) break;
      }
    }
    // phi^{n+1} = phi^(1) / ||phi^(1)||, and max |phi^{n+1} - phi^n|; then one
    // read of the scalars after the last queued iteration, the norm and the change
    if ((st = G.norm(x)) != FSE_OK || (st = G.normalise(x, G.phin, hd)) != FSE_OK) return st;
    cudaError_t e = cudaMemcpyAsync(hs, G.sc, sizeof(double) * SC_SIZE, cudaMemcpyDeviceToHost, G.st);
    if (e != cudaSuccess) return cuda_fail(P, e, "ground state scalars");
    if ((st = G.read(h2, G.out, 2)) != FSE_OK) return st;
    res = hs[SC_RES];
    inner += (int)hs[SC_IT];
    if (!(h2[0] > 0.0)) return fail(P, FSE_ERR_NONFINITE, "ground state: zero field");
    change = h2[1] / o.dt;
    ++outer;
    if (!std::isfinite(change)) return fail(P, FSE_ERR_NONFINITE, "ground state: non-finite iterate");
    if (change <= o.tol) break;
  }
  if (info) {
    info->outer = outer;
    info->inner = (int)std::min<long long>(inner, 0x7fffffff);
    info->change = change;
    info->residual = res;
  }
  return FSE_OK;
}

}  // namespace
}  // namespace fse

using namespace fse;

extern "C" fse_status fse_ground_state_workspace(fse_plan_t P, size_t* bytes) {
  if (!P || !bytes) return FSE_ERR_INVALID;
  *bytes = gs_layout(P).total;
  return FSE_OK;
}

extern "C" fse_status fse_ground_state(fse_plan_t P, void* psi, void* workspace, size_t bytes,
                                       const fse_gs_opts* opts, fse_gs_info* info) {
  if (!P || !psi || !workspace || !opts) return FSE_ERR_INVALID;
  if (!P->ws || !P->precomputed) return fail(P, FSE_ERR_INVALID, "fse_kernel_precompute has not run");
  if (reinterpret_cast<uintptr_t>(psi) % P->csize != 0 || reinterpret_cast<uintptr_t>(workspace) % 256 != 0)
    return fail(P, FSE_ERR_INVALID, "misaligned buffer");
  if (bytes < gs_layout(P).total) return fail(P, FSE_ERR_NOMEM, "ground-state workspace too small");
  if (!(opts->dt > 0.0) || opts->max_outer < 0 || opts->max_inner < 0 || !(opts->tol >= 0.0) ||
      !(opts->inner_tol >= 0.0))
    return fail(P, FSE_ERR_INVALID, "ground state: bad options");
  if (!P->gs_host) {
    void* h = nullptr;
    cudaError_t e = cudaMallocHost(&h, sizeof(double) * 2 * SC_SIZE);
    if (e != cudaSuccess) return cuda_fail(P, e, "ground state host scalars");
    P->gs_host = static_cast<double*>(h);
  }
  for (auto& ev : P->gs_ev) {
    if (ev) continue;
    cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(P, e, "ground state events");
  }
  if (!P->gs_stream) {
    cudaError_t e = cudaStreamCreateWithFlags(&P->gs_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&P->gs_fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&P->gs_join, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(P, e, "ground state stream");
  }
  // the solve runs on a stream of the plan's own (see fse_plan::gs_stream),
  // after and before the caller's stream
  cudaStream_t user = P->stream;
  cudaError_t e = cudaEventRecord(P->gs_fork, user);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(P->gs_stream, P->gs_fork, 0);
  if (e != cudaSuccess) return cuda_fail(P, e, "ground state fork");
  P->stream = P->gs_stream;
  const fse_status st = P->prec == FSE_F32 ? ground_state<float>(P, psi, workspace, *opts, info)
                                           : ground_state<double>(P, psi, workspace, *opts, info);
  P->stream = user;
  e = cudaEventRecord(P->gs_join, P->gs_stream);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(user, P->gs_join, 0);
  if (e == cudaSuccess) e = cudaStreamSynchronize(user);
  if (st == FSE_OK && e != cudaSuccess) return cuda_fail(P, e, "ground state join");
  return st;
}

extern "C" fse_status fse_shift_kick(fse_plan_t P, void* psi, const double* x0, const double* k) {
  if (!P || !psi) return FSE_ERR_INVALID;
  if (!P->ws || !P->precomputed) return fail(P, FSE_ERR_INVALID, "fse_kernel_precompute has not run");
  if (reinterpret_cast<uintptr_t>(psi) % P->csize != 0) return fail(P, FSE_ERR_INVALID, "misaligned buffer");
  for (int j = 0; j < P->dim; ++j)
    if ((x0 && !std::isfinite(x0[j])) || (k && !std::isfinite(k[j])))
      return fail(P, FSE_ERR_INVALID, "shift or kick not finite");
  return P->prec == FSE_F32 ? shift_kick<float>(P, psi, x0, k) : shift_kick<double>(P, psi, x0, k);
}
