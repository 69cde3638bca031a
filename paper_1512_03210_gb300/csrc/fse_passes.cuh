// fse_passes.cuh -- the fused passes of one TS2-GauSum step (Section 4.2, Eqs. tssp1-tssp3).
//
// Data layout in HBM (x fastest, interleaved complex):
//   psi  [nz][ny][nx]            the wave function phi(x~) or its partial spectra
//   S    [nz][2ny][sx] (3D)      x-half-spectrum of the zero-padded density,
//        [ny][sx]      (2D)      sx >= nx+1 (row stride, a multiple of 16)
//   Chat [nz+1][ny+1][nx+1]      kernel transform C^ on |p_j| = 0..n_j (Real)
//
// Passes (3D; 2D drops the z passes and fuses the y passes):
//   X0  fwd-x of psi                                   (start of a call)
//   B   fwd-y of psi                 D  inv-y of psi
//   C   z: fwd . exp(-i f theta_k)/N . inv             (kinetic, Eq. tssp1/tssp3)
//   E   inv-x of psi -> u1 (stored) -> rho=|u1|^2 -> zero-padded R2C along x into S
//   F   y of S: load ny rows, zero-pad to 2ny, fwd
//   G   z of S: load nz rows, zero-pad to 2nz, fwd . K^_n/Npad . inv, keep nz rows
//   H   y of S: inv, keep ny rows
//   A   C2R inv-x of S (crop) -> varphi -> u2 = u1 exp(-i Theta) -> fwd-x of psi
//   XI  inv-x of psi                                   (end of a call)
// Theta = dt beta |u1|^2 + lambda varphi + P_n(x~) (Eqs. solu_step2, int_poten).
#pragma once

#include "fse_col.cuh"

namespace fse {

enum { XP_FWD = 0, XP_INV = 1, XP_E = 2, XP_A = 3, XP_R = 4, XP_ADJ1 = 5, XP_ADJ2 = 6, XP_AL = 7, XP_D = 8, XP_LZ = 9 };

struct XArgs {
  void* psi;
  void* spec;
  int nlines, ny, srow_mul;
  int use_spec;           // pass A: 0 = no nonlocal term (varphi = 0)
  long long sx;
  double beta_dt, lam;
  double pa, pb, pc, pe;  // P = pa x^2 + pb y^2 + pc x y + pe z^2
  double lo0, lo1, lo2, h0, h1, h2;
  double* part;           // pass R: partial of sum varphi |psi|^2; passes E / XI: partial of sum |u1|^2
  const double* scale;    // pass A: optional renormalisation factor (device scalar)
  const void* aux;        // adjoint passes, A: u1 (output of the first kinetic half step); X0: its input
  long long part_stride;  // adjoint pass 1: distance between the three gradient slots
  int ix0;                // adjoint pass 1: the index along x next to the coordinate's zero
  double dp[12];          // adjoint pass 1: dP/dgamma_v = dp[4v] x^2 + dp[4v+1] y^2 + dp[4v+2] x y + dp[4v+3] z^2
  // optical lattice lat_amp sum_v sin^2(lat_k[v] x_v): its integral over the
  // window is sum_q lat_w[q] V_lat(x(tau_q)), x = (c x~ + s y~, -s x~ + c y~, z~)
  // with (c, s) = (lat_c[q], lat_s[q]) = (cos, sin)(Omega tau_q)
  double lat_amp;
  double lat_k[3];
  int lat_nq;
  double lat_w[16], lat_c[16], lat_s[16];
  void* out;              // pass R: optional real array receiving varphi (the nonlocal potential); E, XI: u1
  // float copies of the scalars above (see MulArgs::f)
  struct {
    float beta_dt, lam, pa, pb, pc, pe, lo0, lo1, lo2, h0, h1, h2;
    float lat_amp, lat_k[3], lat_w[16], lat_c[16], lat_s[16];
  } f;
};

__host__ __device__ inline void fill_f32(XArgs& a) {
  a.f.beta_dt = (float)a.beta_dt;
  a.f.lam = (float)a.lam;
  a.f.pa = (float)a.pa;
  a.f.pb = (float)a.pb;
  a.f.pc = (float)a.pc;
  a.f.pe = (float)a.pe;
  a.f.lo0 = (float)a.lo0;
  a.f.lo1 = (float)a.lo1;
  a.f.lo2 = (float)a.lo2;
  a.f.h0 = (float)a.h0;
  a.f.h1 = (float)a.h1;
  a.f.h2 = (float)a.h2;
  a.f.lat_amp = (float)a.lat_amp;
  for (int i = 0; i < 3; ++i) a.f.lat_k[i] = (float)a.lat_k[i];
  for (int i = 0; i < 16; ++i) {
    a.f.lat_w[i] = (float)a.lat_w[i];
    a.f.lat_c[i] = (float)a.lat_c[i];
    a.f.lat_s[i] = (float)a.lat_s[i];
  }
}

// Rounded products and fused multiply-adds that the compiler does not
// re-associate or contract, so that every kernel that inlines an expression
// built from them (the single-run and the batched passes) computes the same bits.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// ---------------------------------------------------------------------------
// x passes over tiles of LN consecutive lines (rows of psi). A group of the
// wave function's transforms (length n) is a pair of lines for float, one line
// for double; the real density is handled as two lines packed into one complex
// line, and a group of its transforms (length 2n, zero-padded or cropped) is
// four lines for float, two for double. Either way a tile holds LP groups of n
// or LP / 2 groups of 2n elements of 16 bytes, worked on by the same LP * T
// threads.
//
// The first pass of every transform takes its inputs straight from global
// memory (positions j + r n/R: consecutive threads read along the line) and the
// last one stores straight back. Real fields (the densities before the R2C,
// the potential after the C2R) cross the tile as plain reals, line by line, so
// that their accesses are free of bank conflicts; only the half spectra, whose
// bins k and 2n - k meet, go through the tile as elements.
// ---------------------------------------------------------------------------
template <typename Real, int NX, int LN_>
struct XCfg {
  typedef typename LaneOf<Real>::T L;
  static constexpr int CW = sizeof(L) / sizeof(Real);  // lines per group of psi
  static constexpr int LN = LN_, LP = LN / CW, LQ = LP / 2;
  typedef FftCfg<Real, NX, 0, true> F1;
  typedef FftCfg<Real, 2 * NX, 2 * F1::T, true> F2;
  static constexpr int T = F1::T, NT = LP * T;
  static constexpr int E = F1::E > F2::E ? F1::E : F2::E;
  static constexpr int MR1 = F1::RF < F1::RL ? F1::RF : F1::RL;
  // line strides of the tile in elements (see XAddr)
  static constexpr int MR2 = F2::RF < F2::RL ? F2::RF : F2::RL;
  static constexpr int LS1 = NX + NX / MR1, LS2 = 2 * NX + 2 * NX / MR2;
  static constexpr int RS = NX + 4;  // line stride of a real field in the tile
  static constexpr size_t B1 = 16 * (size_t)LP * LS1, B2 = 16 * (size_t)LQ * LS2;
  __host__ __device__ static constexpr size_t smem() { return B1 > B2 ? B1 : B2; }
  __host__ __device__ static constexpr int minb() {
    const int thr = E > 12 || (sizeof(Real) == 8 && E > 6) ? 512 : (E > 8 || sizeof(Real) == 8 ? 640 : 1024);
    const int b = thr / ((NT + 31) / 32 * 32);
    return b < 1 ? 1 : (b > 32 ? 32 : b);
  }
};

// Address map of group `base / LS`: an element is skipped after every FR, so
// that the first pass's writes (rows FR apart) fall on different banks.
struct XAddr {
  int base;
  template <int FR> __device__ __forceinline__ int slot(int row) const { return base + row + row / FR; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};

// Lines per tile: 16 (float) or 8 (double) wide, fewer where a line's threads
// are many; narrow tiles fill a warp. float64 lines take T >= 32 threads.
template <typename Real, int NX> struct XWidths {
  static constexpr int CW = XCfg<Real, NX, 16>::CW, T = XCfg<Real, NX, 16>::T;
  __host__ __device__ static constexpr int wide() {
    int lp = 512 / T < 8 ? 512 / T / 2 * 2 : 8;
    if (T >= 64 && sizeof(Real) == 4) lp = 4;
    while (lp * T < 32) lp *= 2;
    return lp * CW;
  }
  __host__ __device__ static constexpr int narrow() {
    int lp = 2;
    while (lp * T < 32) lp *= 2;
    return lp * CW < wide() ? lp * CW : wide();
  }
};

// Rows of S holding the x-half-spectra of a tile's lines (mul * ny rows per z;
// one division per tile rather than one per element).
struct SRows {
  int y0, z0, ny, mul;
  __device__ __forceinline__ SRows(const XArgs& a, int l0) : y0(l0 % a.ny), z0(l0 / a.ny), ny(a.ny), mul(a.srow_mul) {}
  __device__ __forceinline__ long long row(int u) const {
    int y = y0 + u, z = z0;
    while (y >= ny) {
      y -= ny;
      ++z;
    }
    return (long long)z * (mul * ny) + y;
  }
};

// The transformed densities in the tile (element k of group q) -> x-half-spectra
// of the tile's lines in S: A_k = (Z_k + conj Z_-k)/2, B_k = (Z_k - conj Z_-k)/(2i)
// for the two real lines of a complex line. Bins in pairs (2b, 2b + 1), one
// 16-byte store per line (rows of S are 16-byte aligned); the last pair is bin
// NX alone. Ends without a barrier.
template <int NX, int LN>
__device__ __forceinline__ void r2c_separate(const XArgs& a, const float4* buf, int l0, float*) {
  typedef XCfg<float, NX, LN> K;
  constexpr int NB = NX / 2 + 1, FR = K::F2::RF;
  float2* S = reinterpret_cast<float2*>(a.spec);
  const SRows sr(a, l0);
  const float2 half = make_float2(0.5f, 0.5f);
#pragma unroll 2
  for (int idx = threadIdx.x; idx < K::LQ * NB; idx += K::NT) {
    const int q = idx / NB, k0 = 2 * (idx % NB);
    const XAddr ad{q * K::LS2};
    float2 vals[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = min(k0 + h, NX);
      Vec<float2> zk, zm;
      slot_ld(buf, ad.slot<FR>(k), zk);
      slot_ld(buf, ad.slot<FR>(k == 0 ? 0 : 2 * NX - k), zm);
      const float2 ar = lmul(half, ladd(zk.re, zm.re)), ai = lmul(half, lsub(zk.im, zm.im));
      const float2 br = lmul(half, ladd(zk.im, zm.im)), bi = lmul(half, lsub(zm.re, zk.re));
      // lane c of group q carries real lines 4q + 2c (A) and 4q + 2c + 1 (B)
      vals[h][0] = make_float2(ar.x, ai.x);
      vals[h][1] = make_float2(br.x, bi.x);
      vals[h][2] = make_float2(ar.y, ai.y);
      vals[h][3] = make_float2(br.y, bi.y);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int l = l0 + 4 * q + u;
      if (l >= a.nlines) continue;
      float2* row = &S[sr.row(4 * q + u) * a.sx + k0];
      if (k0 < NX)
        *reinterpret_cast<float4*>(row) = make_float4(vals[0][u].x, vals[0][u].y, vals[1][u].x, vals[1][u].y);
      else
        *row = vals[0][u];
    }
  }
}
template <int NX, int LN>
__device__ __forceinline__ void r2c_separate(const XArgs& a, const float4* buf, int l0, double*) {
  typedef XCfg<double, NX, LN> K;
  constexpr int FR = K::F2::RF;
  double2* S = reinterpret_cast<double2*>(a.spec);
  const SRows sr(a, l0);
#pragma unroll 2
  for (int idx = threadIdx.x; idx < K::LQ * (NX + 1); idx += K::NT) {
    const int q = idx / (NX + 1), k = idx % (NX + 1), l = l0 + 2 * q;
    const XAddr ad{q * K::LS2};
    Vec<double> zk, zm;
    slot_ld(buf, ad.slot<FR>(k), zk);
    slot_ld(buf, ad.slot<FR>(k == 0 ? 0 : 2 * NX - k), zm);
    if (l < a.nlines)
      S[sr.row(2 * q) * a.sx + k] = make_double2(0.5 * (zk.re + zm.re), 0.5 * (zk.im - zm.im));
    if (l + 1 < a.nlines)
      S[sr.row(2 * q + 1) * a.sx + k] = make_double2(0.5 * (zk.im + zm.im), 0.5 * (zm.re - zk.re));
  }
}

// x-half-spectra in S of the tile's lines -> elements Z_k = A + i B, Z_{2n-k} =
// conj(A) + i conj(B) of every group in the tile. Ends without a barrier.
template <int NX, int LN>
__device__ __forceinline__ void c2r_gather(const XArgs& a, float4* buf, int l0, float*) {
  typedef XCfg<float, NX, LN> K;
  constexpr int NB = NX / 2 + 1, FR = K::F2::RF;
  const float2* S = reinterpret_cast<const float2*>(a.spec);
  const SRows sr(a, l0);
#pragma unroll 2
  for (int idx = threadIdx.x; idx < K::LQ * NB; idx += K::NT) {
    const int q = idx / NB, k0 = 2 * (idx % NB);
    const XAddr ad{q * K::LS2};
    float4 v[4];
    // the last pair holds bin NX and a padding bin of the row, which is not used
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int l = l0 + 4 * q + u;
      v[u] = l < a.nlines ? *reinterpret_cast<const float4*>(&S[sr.row(4 * q + u) * a.sx + k0])
                          : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = k0 + h;
      if (k > NX) break;
      float2 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = h ? make_float2(v[u].z, v[u].w) : make_float2(v[u].x, v[u].y);
      const Vec<float2> zk{make_float2(w[0].x - w[1].y, w[2].x - w[3].y), make_float2(w[0].y + w[1].x, w[2].y + w[3].x)};
      slot_st(buf, ad.slot<FR>(k), zk);
      if (k > 0 && k < NX) {
        const Vec<float2> zm{make_float2(w[0].x + w[1].y, w[2].x + w[3].y), make_float2(w[1].x - w[0].y, w[3].x - w[2].y)};
        slot_st(buf, ad.slot<FR>(2 * NX - k), zm);
      }
    }
  }
}
template <int NX, int LN>
__device__ __forceinline__ void c2r_gather(const XArgs& a, float4* buf, int l0, double*) {
  typedef XCfg<double, NX, LN> K;
  constexpr int FR = K::F2::RF;
  const double2* S = reinterpret_cast<const double2*>(a.spec);
  const SRows sr(a, l0);
#pragma unroll 2
  for (int idx = threadIdx.x; idx < K::LQ * (NX + 1); idx += K::NT) {
    const int q = idx / (NX + 1), k = idx % (NX + 1), l = l0 + 2 * q;
    const XAddr ad{q * K::LS2};
    double2 A = make_double2(0.0, 0.0), B = A;
    if (l < a.nlines) A = S[sr.row(2 * q) * a.sx + k];
    if (l + 1 < a.nlines) B = S[sr.row(2 * q + 1) * a.sx + k];
    slot_st(buf, ad.slot<FR>(k), Vec<double>{A.x - B.y, A.y + B.x});
    if (k > 0 && k < NX) slot_st(buf, ad.slot<FR>(2 * NX - k), Vec<double>{A.x + B.y, B.x - A.y});
  }
}

// A real field of the tile's lines, line l at row l (RS reals apart): values of
// a group's lines at one position. psi groups (CW lines) and density groups (2 CW).
template <int RS> __device__ __forceinline__ void real_st(float* f, int g, int x, float2 v) {
  f[(2 * g) * RS + x] = v.x;
  f[(2 * g + 1) * RS + x] = v.y;
}
template <int RS> __device__ __forceinline__ void real_st(double* f, int g, int x, double v) { f[g * RS + x] = v; }
template <int RS> __device__ __forceinline__ void real_ld(const float* f, int g, int x, float2& v) {
  v = make_float2(f[(2 * g) * RS + x], f[(2 * g + 1) * RS + x]);
}
template <int RS> __device__ __forceinline__ void real_ld(const double* f, int g, int x, double& v) { v = f[g * RS + x]; }
// density group q: lane c = lines 2c (re) and 2c + 1 (im)
template <int RS> __device__ __forceinline__ void real_ld2(const float* f, int q, int x, Vec<float2>& v) {
  const float* p = f + 4 * q * RS + x;
  v = {make_float2(p[0], p[2 * RS]), make_float2(p[RS], p[3 * RS])};
}
template <int RS> __device__ __forceinline__ void real_ld2(const double* f, int q, int x, Vec<double>& v) {
  v = {f[2 * q * RS + x], f[(2 * q + 1) * RS + x]};
}
template <int RS> __device__ __forceinline__ void real_st2(float* f, int q, int x, const Vec<float2>& v) {
  float* p = f + 4 * q * RS + x;
  p[0] = v.re.x;
  p[RS] = v.im.x;
  p[2 * RS] = v.re.y;
  p[3 * RS] = v.im.y;
}
template <int RS> __device__ __forceinline__ void real_st2(double* f, int q, int x, const Vec<double>& v) {
  f[2 * q * RS + x] = v.re;
  f[(2 * q + 1) * RS + x] = v.im;
}

// Elements of a psi group (its lines side by side, nl of the tile's lines from line0 on exist).
template <int NX> __device__ __forceinline__ Vec<float2> line_ld(const float2* line0, int g, int nl, int x) {
  const float2 z = make_float2(0.f, 0.f);
  const float2 u0 = 2 * g < nl ? line0[(2 * g) * NX + x] : z;
  const float2 u1 = 2 * g + 1 < nl ? line0[(2 * g + 1) * NX + x] : z;
  return {make_float2(u0.x, u1.x), make_float2(u0.y, u1.y)};
}
template <int NX> __device__ __forceinline__ void line_st(float2* line0, int g, int nl, int x, const Vec<float2>& u) {
  if (2 * g < nl) line0[(2 * g) * NX + x] = make_float2(u.re.x, u.im.x);
  if (2 * g + 1 < nl) line0[(2 * g + 1) * NX + x] = make_float2(u.re.y, u.im.y);
}
template <int NX> __device__ __forceinline__ Vec<double> line_ld(const double2* line0, int g, int nl, int x) {
  if (g >= nl) return {0.0, 0.0};
  const double2 u = line0[g * NX + x];
  return {u.x, u.y};
}
template <int NX> __device__ __forceinline__ void line_st(double2* line0, int g, int nl, int x, const Vec<double>& u) {
  if (g < nl) line0[g * NX + x] = make_double2(u.re, u.im);
}
__device__ __forceinline__ double lane_sum(float2 v) { return (double)v.x + (double)v.y; }
__device__ __forceinline__ double lane_sum(double v) { return v; }

// cos(th) - 1 and sin(th) for |th| <= 1/2 by their Taylor series (truncation
// below 3e-10 for float, 1e-18 for double) in Horner form.
__device__ __forceinline__ void small_sincos(float2 th, float2& sn, float2& cm1) {
  const float2 t2 = lmul(th, th);
  const float2 ps = lmul(t2, lfma(t2, lfma(t2, lfma(t2, lbc<float2>(1.0 / 362880), lbc<float2>(-1.0 / 5040)), lbc<float2>(1.0 / 120)),
                                  lbc<float2>(-1.0 / 6)));
  cm1 = lmul(t2, lfma(t2, lfma(t2, lfma(t2, lbc<float2>(1.0 / 40320), lbc<float2>(-1.0 / 720)), lbc<float2>(1.0 / 24)),
                      lbc<float2>(-0.5)));
  sn = lfma(th, ps, th);
}
__device__ __forceinline__ void small_sincos(double th, double& sn, double& cm1) {
  const double t2 = th * th;
  double s = -1.0 / 1307674368000.0, c = -1.0 / 87178291200.0;
  s = lfma(s, t2, 1.0 / 6227020800.0);
  c = lfma(c, t2, 1.0 / 479001600.0);
  s = lfma(s, t2, -1.0 / 39916800.0);
  c = lfma(c, t2, -1.0 / 3628800.0);
  s = lfma(s, t2, 1.0 / 362880.0);
  c = lfma(c, t2, 1.0 / 40320.0);
  s = lfma(s, t2, -1.0 / 5040.0);
  c = lfma(c, t2, -1.0 / 720.0);
  s = lfma(s, t2, 1.0 / 120.0);
  c = lfma(c, t2, 1.0 / 24.0);
  s = lfma(s, t2, -1.0 / 6.0);
  c = lfma(c, t2, -0.5);
  cm1 = c * t2;
  sn = lfma(th, s * t2, th);
}

// u exp(-i th). For |th| <= 1/2 the product is u + u (cos th - 1 - i sin th),
// whose second summand is small: the factor's modulus is then off by no more
// than |th|^2 times the rounding unit, with no steady drift of the norm. Larger
// phases go through sincos, the pair's modulus error folded into the products
// (unit_mul).
__device__ __forceinline__ Vec<float2> phase_mul(const Vec<float2>& u, float2 th) {
  if (fmaxf(fabsf(th.x), fabsf(th.y)) <= 0.5f) {
    float2 s, c;
    small_sincos(th, s, c);
    return {ladd(u.re, lfma(u.re, c, lmul(u.im, s))), ladd(u.im, lfma(u.im, c, lneg(lmul(u.re, s))))};
  }
  float s0, c0, s1, c1;
  sincosf(th.x, &s0, &c0);
  sincosf(th.y, &s1, &c1);
  const float2 a = unit_mul(make_float2(u.re.x, u.im.x), c0, -s0, false);
  const float2 b = unit_mul(make_float2(u.re.y, u.im.y), c1, -s1, false);
  return {make_float2(a.x, b.x), make_float2(a.y, b.y)};
}
__device__ __forceinline__ Vec<double> phase_mul(const Vec<double>& u, double th) {
  double s, c;
  if (fabs(th) <= 0.5) {
    small_sincos(th, s, c);
    c += 1.0;
  } else {
    sincos(th, &s, &c);
  }
  return {lfma(u.re, c, lmul(u.im, s)), lfma(u.im, c, lmul(u.re, -s))};
}

template <typename Real>
__device__ __forceinline__ Real sin_sq(Real v);
template <> __device__ __forceinline__ float sin_sq(float v) {
  const float s = sinf(v);
  return s * s;
}
template <> __device__ __forceinline__ double sin_sq(double v) {
  const double s = sin(v);
  return s * s;
}

// Window integral of the optical lattice at the point (X, Y, Z) of the rotating
// frame (Gauss-Legendre nodes of the window in a.lat_*).
template <typename Real>
__device__ __forceinline__ Real lattice_integral(const XArgs& a, Real X, Real Y, Real Z) {
  const Real kx = prm<Real>(a.lat_k[0], a.f.lat_k[0]), ky = prm<Real>(a.lat_k[1], a.f.lat_k[1]);
  const Real kz = prm<Real>(a.lat_k[2], a.f.lat_k[2]);
  const Real zt = kz != Real(0) ? sin_sq(kz * Z) : Real(0);
  Real acc = Real(0);
  for (int q = 0; q < a.lat_nq; ++q) {
    const Real c = prm<Real>(a.lat_c[q], a.f.lat_c[q]), s = prm<Real>(a.lat_s[q], a.f.lat_s[q]);
    const Real xr = c * X + s * Y, yr = -s * X + c * Y;
    acc += prm<Real>(a.lat_w[q], a.f.lat_w[q]) * (sin_sq(kx * xr) + sin_sq(ky * yr) + zt);
  }
  return prm<Real>(a.lat_amp, a.f.lat_amp) * acc;
}
// The same for the lanes' points of one x, the nodes' sines of all lanes in one
// loop.
template <typename Real, int CW>
__device__ __forceinline__ void lattice_lanes(const XArgs& a, Real X, const Real (&Y)[CW], const Real (&Z)[CW], Real (&out)[CW]) {
  const Real kx = prm<Real>(a.lat_k[0], a.f.lat_k[0]), ky = prm<Real>(a.lat_k[1], a.f.lat_k[1]);
  const Real kz = prm<Real>(a.lat_k[2], a.f.lat_k[2]);
  Real zt[CW], acc[CW];
#pragma unroll
  for (int l = 0; l < CW; ++l) {
    zt[l] = kz != Real(0) ? sin_sq(kz * Z[l]) : Real(0);
    acc[l] = Real(0);
  }
#pragma unroll 1
  for (int q = 0; q < a.lat_nq; ++q) {
    const Real c = prm<Real>(a.lat_c[q], a.f.lat_c[q]), s = prm<Real>(a.lat_s[q], a.f.lat_s[q]);
    const Real w = prm<Real>(a.lat_w[q], a.f.lat_w[q]);
#pragma unroll
    for (int l = 0; l < CW; ++l) {
      const Real xr = c * X + s * Y[l], yr = -s * X + c * Y[l];
      acc[l] += w * (sin_sq(kx * xr) + sin_sq(ky * yr) + zt[l]);
    }
  }
#pragma unroll
  for (int l = 0; l < CW; ++l) out[l] = prm<Real>(a.lat_amp, a.f.lat_amp) * acc[l];
}
// out of line, for the adjoint's unrolled loop (the arguments go through local memory)
template <typename Real>
__device__ __noinline__ Real lattice_call(const XArgs& a, Real X, Real Y, Real Z) {
  return lattice_integral<Real>(a, X, Y, Z);
}


// This thread's lines: the trap's window integral on them is P = (pa X + cy) X + c0
// (harmonic quadratic form) plus the optical lattice.
template <typename Real, int CW> struct LineTrap {
  typedef typename LaneOf<Real>::T L;
  Real Y[CW], Z[CW];
  L cy, c0;
};
template <typename Real, int CW>
__device__ __forceinline__ LineTrap<Real, CW> line_trap(const XArgs& a, int l) {
  LineTrap<Real, CW> t;
  Real cy[CW], c0[CW];
#pragma unroll
  for (int q = 0; q < CW; ++q) {
    const int y = (l + q) % a.ny, z = (l + q) / a.ny;
    t.Y[q] = fma_rn(prm<Real>(a.h1, a.f.h1), Real(y), prm<Real>(a.lo1, a.f.lo1));
    t.Z[q] = fma_rn(prm<Real>(a.h2, a.f.h2), Real(z), prm<Real>(a.lo2, a.f.lo2));
    cy[q] = mul_rn(prm<Real>(a.pc, a.f.pc), t.Y[q]);
    c0[q] = fma_rn(mul_rn(prm<Real>(a.pe, a.f.pe), t.Z[q]), t.Z[q], mul_rn(mul_rn(prm<Real>(a.pb, a.f.pb), t.Y[q]), t.Y[q]));
  }
  t.cy = lane_of(cy);
  t.c0 = lane_of(c0);
  return t;
}
template <typename Real, int CW, bool LAT>
__device__ __forceinline__ typename LaneOf<Real>::T trap_phase(const XArgs& a, const LineTrap<Real, CW>& t, int x, bool lat) {
  typedef typename LaneOf<Real>::T L;
  const Real X = fma_rn(prm<Real>(a.h0, a.f.h0), Real(x), prm<Real>(a.lo0, a.f.lo0));
  const L Xb = lbc<L>(X);
  L P = lfma(lfma(lbc<L>(prm<Real>(a.pa, a.f.pa)), Xb, t.cy), Xb, t.c0);
  if (LAT && lat) {
    Real v[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q) v[q] = lattice_call<Real>(a, X, t.Y[q], t.Z[q]);
    P = ladd(P, lane_of(v));
  }
  return P;
}
__device__ __forceinline__ float lane_get(float2 v, int q) { return q ? v.y : v.x; }
__device__ __forceinline__ double lane_get(double v, int) { return v; }

// Pass A with a lattice (XP_AL) keeps the lattice's window integrals of a tile's
// points in shared memory, line by line behind the tile. They depend on nothing
// that an earlier pass writes and are formed first, while nothing else is live,
// in narrow tiles by warps that only come for this and leave: the 32 threads of
// an 8 x 8 or 12 x 8 grid's tile took 13 and 61 us over them. Calls of two steps:
// 8 x 8 43 -> 28 us, 12 x 8 float64 143 -> 62, 96 x 128 88 -> 56, 512^2 109 -> 86,
// 128 x 192 x 24 247 -> 154, 512^2 float64 (its sines) 935 -> 913.
template <typename Real, int NX, int LN, int KIND> struct XLaunch {
  typedef XCfg<Real, NX, LN> K;
  static constexpr bool LAT = KIND == XP_AL, HELP = LAT && LN == XWidths<Real, NX>::narrow();
  static constexpr int threads = HELP && K::NT < 256 ? 256 : K::NT;
  __host__ __device__ static constexpr size_t smem() { return K::smem() + (LAT ? sizeof(Real) * (size_t)LN * K::RS : 0); }
  __host__ __device__ static constexpr int minb() { return HELP ? 2 : K::minb(); }
};

// PDL: the launch is a dependent one (the prologue's wait is here).
template <typename Real, int NX, int LN, int KIND, bool PDL>
__device__ __forceinline__ void xpass_body(const XArgs& a, const typename TwOf<Real>::T* __restrict__ twn,
                                           const typename TwOf<Real>::T* __restrict__ tw2n, int bid) {
  typedef XCfg<Real, NX, LN> K;
  typedef typename K::F1 F1;
  typedef typename K::F2 F2;
  typedef typename Cplx<Real>::T C;
  typedef typename K::L L;
  constexpr int CW = K::CW, T = K::T, RS = K::RS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  float4* buf = reinterpret_cast<float4*>(smem_raw);
  Real* field = reinterpret_cast<Real*>(smem_raw);
  const int tid = threadIdx.x;
  int it = tid % T;
  const int g = tid / T;                            // psi group and item
  int it2 = tid % (2 * T);
  const int q2 = tid / (2 * T);                     // density group and item
  const XAddr ad1{g * K::LS1}, ad2{q2 * K::LS2};
  const int l0 = bid * LN, nl = a.nlines - l0;
  C* line0 = reinterpret_cast<C*>(a.psi) + (long long)l0 * NX;
  Real* lat = reinterpret_cast<Real*>(smem_raw + K::smem());
  if constexpr (KIND == XP_AL) {
    typedef XLaunch<Real, NX, LN, KIND> X;
#pragma unroll 1
    for (int i = tid; i < K::LP * NX; i += X::threads) {
      const int h = i / NX, x = i - h * NX;
      Real Y[CW], Z[CW], v[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) {
        const int l = l0 + CW * h + q;
        Y[q] = fma_rn(prm<Real>(a.h1, a.f.h1), Real(l % a.ny), prm<Real>(a.lo1, a.f.lo1));
        Z[q] = fma_rn(prm<Real>(a.h2, a.f.h2), Real(l / a.ny), prm<Real>(a.lo2, a.f.lo2));
      }
      lattice_lanes<Real, CW>(a, fma_rn(prm<Real>(a.h0, a.f.h0), Real(x), prm<Real>(a.lo0, a.f.lo0)), Y, Z, v);
      real_st<RS>(lat, h, x, lane_of(v));
    }
    __syncthreads();
    if (X::threads > K::NT && tid >= K::NT) return;
  }
  if constexpr (PDL && LN == XWidths<Real, NX>::narrow() && LN < XWidths<Real, NX>::wide()) {
    // a narrow tile is alone on its SM: its twiddle tables come into L1 before
    // the wait for the previous pass (see col_tile)
    unsigned x = 0;
    if constexpr (KIND != XP_R && KIND != XP_ADJ1 && KIND != XP_ADJ2 && KIND != XP_D)
      x = F1::template warm_table<false, true, K::NT>(twn, tid);
    if constexpr (KIND != XP_FWD && KIND != XP_INV) {
      if (KIND == XP_LZ) x ^= F1::template warm_table<true, true, K::NT>(twn, tid);
      if (KIND == XP_E || KIND == XP_D || (KIND == XP_ADJ1 && a.use_spec)) x ^= F2::template warm_table<false, false, K::NT>(tw2n, tid);
      if (KIND != XP_E && KIND != XP_D && KIND != XP_LZ && a.use_spec) x ^= F2::template warm_table<true, false, K::NT>(tw2n, tid);
    }
    reinterpret_cast<unsigned*>(smem_raw)[tid] = x;
  }
  if constexpr (PDL) pass_prologue();
  if constexpr (PDL && LN == XWidths<Real, NX>::narrow() && LN < XWidths<Real, NX>::wide())
    __syncthreads();  // the warm-up's words are written before the tile is
  // hides that the items are unchanged, so that addresses are computed again
  // rather than held in registers across a whole transform
  auto fresh = [&]() { asm volatile("" : "+r"(it), "+r"(it2)); };

  // densities (or other real fields) in `field` -> x-half-spectra of the zero-padded lines in S
  auto r2c = [&]() {
    Vec<L> z[F2::E];
    F2::template each<F2::RF>(it2, [&](int e, int row, int r) {
      if (2 * r < F2::RF) real_ld2<RS>(field, q2, row, z[e]);
    });
    F2::template run<-1, false, false, true, true>(z, buf, ad2, tw2n, it2);
    __syncthreads();
    F2::template each<F2::RL>(it2, [&](int e, int row, int) { slot_st(buf, ad2.template slot<F2::RF>(row), z[e]); });
    __syncthreads();
    r2c_separate<NX, LN>(a, buf, l0, (Real*)nullptr);
  };
  // x-half-spectra in S -> the cropped real field in `field` (ends with a barrier)
  auto c2r = [&]() {
    c2r_gather<NX, LN>(a, buf, l0, (Real*)nullptr);
    __syncthreads();
    Vec<L> z[F2::E];
    F2::template each<F2::RL>(it2, [&](int e, int row, int) { slot_ld(buf, ad2.template slot<F2::RF>(row), z[e]); });
    // radices in reverse: the rows kept by the crop are outputs r < RF/2 of every item
    F2::template run<+1, false, true, true>(z, buf, ad2, tw2n, it2);
    __syncthreads();
    F2::template each<F2::RF>(it2, [&](int e, int row, int r) {
      if (2 * r < F2::RF) real_st2<RS>(field, q2, row, z[e]);
    });
    __syncthreads();
  };

  if constexpr (KIND == XP_D) {
    // the density of psi itself (psi is only read)
    F1::template each<F1::RF>(it, [&](int, int x, int) {
      const Vec<L> u = line_ld<NX>((const C*)line0, g, nl, x);
      real_st<RS>(field, g, x, lfma(u.re, u.re, lmul(u.im, u.im)));
    });
    __syncthreads();
    r2c();
  } else if constexpr (KIND == XP_LZ) {
    // partial of -sum y Im(conj(psi) d_x psi), d_x by the line's own transforms (beta_dt: 2 pi / (W n))
    Vec<L> v[F1::E];
    F1::template each<F1::RF>(it, [&](int e, int x, int) { v[e] = line_ld<NX>((const C*)line0, g, nl, x); });
    const float um = vmax_abs<F1>(it, v);
    F1::template run<-1, true, false, false>(v, buf, ad1, twn, it);
    const Real dk = prm<Real>(a.beta_dt, a.f.beta_dt);
    F1::template each<F1::RL>(it, [&](int e, int k, int) {
      // the odd factor is zero at the Nyquist index
      const L kk = lbc<L>(2 * k == NX ? Real(0) : dk * Real(wrap_index(k, NX)));
      v[e] = {lneg(lmul(kk, v[e].im)), lmul(kk, v[e].re)};
    });
    F1::template run<+1, true, true, true>(v, buf, ad1, twn, it);
    fresh();
    const Pow2<L> su = pow2_scale<L>(um), sd = pow2_scale<L>(vmax_abs<F1>(it, v));
    ExactSum<L> s;
    F1::template each<F1::RF>(it, [&](int e, int x, int) {
      lz_add(line_ld<NX>((const C*)line0, g, nl, x), v[e], su.scale, sd.scale, s);
    });
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < CW; ++q) t -= (a.lo1 + a.h1 * ((l0 + CW * g + q) % a.ny)) * s.get(q);
    t *= su.inv * sd.inv;
    t = block_sum(t, red);
    if (tid == 0) a.part[bid] = t;
  } else if constexpr (KIND == XP_FWD || KIND == XP_INV || KIND == XP_E) {
    Vec<L> v[F1::E];
    // X0 may read another field than the one it writes (aux), E and XI may write another (out)
    const C* src = (KIND == XP_FWD && a.aux) ? reinterpret_cast<const C*>(a.aux) + (long long)l0 * NX : line0;
    F1::template each<F1::RF>(it, [&](int e, int x, int) { v[e] = line_ld<NX>(src, g, nl, x); });
    F1::template run<(KIND == XP_FWD ? -1 : +1), true, false, false>(v, buf, ad1, twn, it);
    fresh();
    if constexpr (KIND == XP_E) __syncthreads();
    C* dst = (KIND != XP_FWD && a.out) ? reinterpret_cast<C*>(a.out) + (long long)l0 * NX : line0;
    F1::template each<F1::RL>(it, [&](int e, int x, int) {
      line_st<NX>(dst, g, nl, x, v[e]);
      if constexpr (KIND == XP_E) real_st<RS>(field, g, x, lfma(v[e].re, v[e].re, lmul(v[e].im, v[e].im)));
    });
    if constexpr (KIND != XP_FWD) {
      if (a.part) {
        // float64 mass partial of this tile (renormalisation). In a loop of its
        // own: predicated off inside the one above, its float64 instructions
        // would still take their slots on the narrow FP64 pipe.
        double mass = 0.0;
        F1::template each<F1::RL>(it, [&](int e, int, int) {
          mass += lane_sum(lfma(v[e].re, v[e].re, lmul(v[e].im, v[e].im)));
        });
        mass = block_sum(mass, red);
        if (tid == 0) a.part[bid] = mass;
      }
    }
    if constexpr (KIND == XP_E) {
      __syncthreads();
      fresh();
      r2c();
    }
  } else {
    if ((KIND == XP_A || KIND == XP_AL) && tid == 0 && nl > 0 && (reinterpret_cast<uintptr_t>(a.psi) & 15) == 0) {
      // the tile's rows of psi (contiguous) move to L2 while the C2R runs (the
      // bulk prefetch needs a 16-byte aligned start; psi may be only
      // element-aligned, and every line then starts 16-byte aligned too)
      if (!a.aux) prefetch_l2_bulk(line0, (unsigned)(min(LN, nl) * NX * sizeof(C)));
    }
    if (a.use_spec) c2r();
    fresh();
    auto phi_at = [&](int x) {
      L p = lbc<L>(0.0);
      if (a.use_spec) real_ld<RS>(field, g, x, p);
      return p;
    };
    if constexpr (KIND == XP_R) {
      // varphi itself, as a real field in the layout of psi, and (or) the sum
      // over the tile of varphi |psi|^2 (nonlocal interaction energy density)
      Real* phi = reinterpret_cast<Real*>(a.out);
      if (phi) {
        F1::template each<F1::RF>(it, [&](int, int x, int) {
          const L p = phi_at(x);
#pragma unroll
          for (int q = 0; q < CW; ++q)
            if (CW * g + q < nl) phi[(long long)(l0 + CW * g + q) * NX + x] = lane_get(p, q);
        });
      }
      if (!a.part) return;
      float pm = 0.f;
      Vec<L> u[F1::E];
      F1::template each<F1::RF>(it, [&](int e, int x, int) {
        u[e] = line_ld<NX>((const C*)line0, g, nl, x);
        pm = lmax_abs(pm, phi_at(x));
      });
      const Pow2<L> su = pow2_scale<L>(vmax_abs<F1>(it, u)), sp = pow2_scale<L>(pm);
      ExactSum<L> sum;
      F1::template each<F1::RF>(it, [&](int e, int x, int) {
        sum.dens(lmul(sp.scale, phi_at(x)), lmul(su.scale, u[e].re), lmul(su.scale, u[e].im));
      });
      double acc = 0.0;
#pragma unroll
      for (int q = 0; q < CW; ++q)
        if (CW * g + q < nl) acc += sum.get(q);
      acc *= sp.inv * (su.inv * su.inv);
      acc = block_sum(acc, red);
      if (tid == 0) a.part[bid] = acc;
    } else if constexpr (KIND == XP_ADJ2) {
      // adjoint, second half: g_u1 = h + 2 q u1, q = dt beta r + lambda Kc r, r = Im(conj(h) u1)
      const C* u1 = reinterpret_cast<const C*>(a.aux) + (long long)l0 * NX;
      const L bd = lbc<L>(prm<Real>(a.beta_dt, a.f.beta_dt)), lam = lbc<L>(prm<Real>(a.lam, a.f.lam));
      F1::template each<F1::RF>(it, [&](int, int x, int) {
        const Vec<L> u = line_ld<NX>(u1, g, nl, x), h = line_ld<NX>((const C*)line0, g, nl, x);
        const L r = lfma(h.re, u.im, lneg(lmul(h.im, u.re)));
        const L t = lfma(bd, r, lmul(lam, phi_at(x)));
        const L t2 = ladd(t, t);
        line_st<NX>(line0, g, nl, x, Vec<L>{lfma(t2, u.re, h.re), lfma(t2, u.im, h.im)});
      });
    } else {
      const LineTrap<Real, CW> trap = line_trap<Real, CW>(a, l0 + CW * g);
      const L bd = lbc<L>(prm<Real>(a.beta_dt, a.f.beta_dt)), lam = lbc<L>(prm<Real>(a.lam, a.f.lam));
      if constexpr (KIND == XP_ADJ1) {
        // adjoint, first half: g_u2 (in psi) -> h = exp(+i Theta) g_u2 (stored in psi),
        // r = Im(conj(g_u2) u2) -> x-half-spectra of r in S, trap-gradient partials
        const C* u1 = reinterpret_cast<const C*>(a.aux) + (long long)l0 * NX;
        const bool lat = a.lat_amp != 0.0;
        L rr[F1::E];
        F1::template each<F1::RF>(it, [&](int e, int x, int) {
          const Vec<L> u = line_ld<NX>(u1, g, nl, x), gu = line_ld<NX>((const C*)line0, g, nl, x);
          const L rho = lfma(u.re, u.re, lmul(u.im, u.im));
          const L th = lfma(bd, rho, lfma(lam, phi_at(x), trap_phase<Real, CW, true>(a, trap, x, lat)));
          const Vec<L> u2 = phase_mul(u, th);
          const L r = lfma(gu.re, u2.im, lneg(lmul(gu.im, u2.re)));
          rr[e] = r;
          line_st<NX>(line0, g, nl, x, phase_mul(gu, lneg(th)));
        });
        if (a.part) {
          // sums over the thread's part of its lines of r, r X and r X^2, by
          // those of r, r i and r i^2 with i the index from the one next to X = 0
          // (from the grid's middle the terms cancel in a box to one side of zero:
          // 1e-14 of the gradient for a cloud at 0.5 in [0, 16])
          float rm = 0.f;
          F1::template each<F1::RF>(it, [&](int e, int, int) { rm = lmax_abs(rm, rr[e]); });
          const Pow2<L> sr = pow2_scale<L>(rm);
          ExactSum<L> e0, e1, e2;
          F1::template each<F1::RF>(it, [&](int e, int x, int) {
            const L r = lmul(sr.scale, rr[e]);
            const Real i = Real(x - a.ix0);
            e0.add(r);
            e1.prod(r, lane_bc<L>(i));
            e2.prod(r, lane_bc<L>(i * i));
          });
          const double xc = a.lo0 + a.h0 * a.ix0;
          double s0[CW], s1[CW], s2[CW];
#pragma unroll
          for (int q = 0; q < CW; ++q) {
            const double i1 = a.h0 * (sr.inv * e1.get(q)), i2 = a.h0 * a.h0 * (sr.inv * e2.get(q));
            s0[q] = sr.inv * e0.get(q);
            s1[q] = fma(xc, s0[q], i1);
            s2[q] = fma(xc, s1[q] + i1, i2);
          }
          // dP/dgamma_v = dp[4v] X^2 + dp[4v+1] Y^2 + dp[4v+2] X Y + dp[4v+3] Z^2
          double dg[3] = {0.0, 0.0, 0.0};
#pragma unroll
          for (int q = 0; q < CW; ++q) {
            const int l = l0 + CW * g + q;
            const double Y = a.lo1 + a.h1 * (l % a.ny), Z = a.lo2 + a.h2 * (l / a.ny);
#pragma unroll
            for (int v = 0; v < 3; ++v)
              dg[v] += a.dp[4 * v] * s2[q] + (a.dp[4 * v + 1] * Y * Y + a.dp[4 * v + 3] * Z * Z) * s0[q] +
                       a.dp[4 * v + 2] * Y * s1[q];
          }
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            const double d = block_sum(dg[v], red);
            if (tid == 0) a.part[v * a.part_stride + bid] = d;
          }
        }
        if (a.use_spec) {
          __syncthreads();
          F1::template each<F1::RF>(it, [&](int e, int x, int) { real_st<RS>(field, g, x, rr[e]); });
          __syncthreads();
          fresh();
          r2c();
        }
      } else {
        // XP_A / XP_AL: u2 = u1 exp(-i Theta) on the inputs of the forward transform's first pass.
        // The optional renormalisation factor is read and converted once per
        // thread: a conversion from double issues on the narrow FP64 pipe.
        const bool rescale = a.scale != nullptr;
        const L fsc = lbc<L>(rescale ? Real(*a.scale) : Real(1));
        // u1 lies in psi, or in another field (aux)
        const C* u1 = a.aux ? reinterpret_cast<const C*>(a.aux) + (long long)l0 * NX : (const C*)line0;
        Vec<L> v[F1::E];
        F1::template each<F1::RF>(it, [&](int e, int x, int) { v[e] = line_ld<NX>(u1, g, nl, x); });
        F1::template each<F1::RF>(it, [&](int e, int x, int) {
          const Vec<L> u = v[e];
          const L rho = lfma(u.re, u.re, lmul(u.im, u.im));
          L P = trap_phase<Real, CW, false>(a, trap, x, true);
          if constexpr (KIND == XP_AL) {
            L w;
            real_ld<RS>(lat, g, x, w);
            P = ladd(P, w);
          }
          const L th = lfma(bd, rho, lfma(lam, phi_at(x), P));
          v[e] = phase_mul(u, th);
          if (rescale) v[e] = {lmul(fsc, v[e].re), lmul(fsc, v[e].im)};
        });
        fresh();
        F1::template run<-1, true, false, true>(v, buf, ad1, twn, it);
        fresh();
        F1::template each<F1::RL>(it, [&](int e, int x, int) { line_st<NX>(line0, g, nl, x, v[e]); });
      }
    }
  }
}

template <typename Real, int NX, int LN, int KIND>
__global__ void __launch_bounds__(XLaunch<Real, NX, LN, KIND>::threads, XLaunch<Real, NX, LN, KIND>::minb())
k_xpass(XArgs a, const typename TwOf<Real>::T* __restrict__ twn, const typename TwOf<Real>::T* __restrict__ tw2n) {
  xpass_body<Real, NX, LN, KIND, true>(a, twn, tw2n, blockIdx.x);
}

// Lines per tile of the x passes: wide tiles where they give every SM one,
// narrow ones otherwise. The kinds XI, E, R and ADJ1 write one partial per tile.
template <typename Real, int NX> inline int xpass_pick(int nlines, int runs) {
  typedef XWidths<Real, NX> W;
  return (long long)((nlines + W::wide() - 1) / W::wide()) * runs >= kSMs ? W::wide() : W::narrow();
}

// Host-side launchers (explicitly instantiated per precision and kind).
template <typename Real, int KIND>
cudaError_t launch_xpass(int nx, const XArgs& a, const void* twn, const void* tw2n, cudaStream_t st);
// Tiles of an x pass over nlines lines of nx points.
template <typename Real> int xpass_tiles(int nx, int nlines);

}  // namespace fse
