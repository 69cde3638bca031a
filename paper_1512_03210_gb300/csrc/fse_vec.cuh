// fse_vec.cuh -- register DFTs and register-staged Stockham transforms on 16-byte elements.
//
// Every transform of the library works on elements Vec<L> = {re, im} of 16
// bytes: for float64 plans L = double (one column or line), for float32 plans
// L = float2 (a pair of neighbouring columns or lines that see the same rows
// and twiddles, so that each operation is one packed two-lane instruction of
// the sm_100 family). Multiplying by +-i only renames re and im.
//
// A transform of length N runs as two or three passes of large radices
// (FftPlan; 256 = 16 x 16, 128 = 16 x 8, 96 = 12 x 8, 512 = 8 x 8 x 8): the
// first pass's inputs come from the caller in registers, the last pass's
// outputs stay there, and between two passes the tile is exchanged through
// shared memory once. Few large passes are what the float32 passes need: they
// are bound by instruction issue and by the barriers and shared-memory round
// trips of the exchanges, and 16 x 16 has one exchange and 15/16 twiddles per
// element where 8 x 8 x 4 has two and 26/16 (256^3 kinetic pass: 60 M -> 43 M
// warp instructions, 99 -> 82 us).
//
// EXACT transforms (those of the wave function) multiply by head + tail pairs
// of every twiddle and irrational constant: a rounded float pair alone has
// |w| = 1 + O(1e-8), fixed per table entry, and the norm would drift by it in
// every step. Transforms of the density spectrum (which only sets a phase)
// use the head alone. For float64 the two are the same.
#pragma once

#include "fse_fft.cuh"

namespace fse {

// ---------------------------------------------------------------------------
// lanes
// ---------------------------------------------------------------------------
template <typename Real> struct LaneOf;
template <> struct LaneOf<float> { typedef float2 T; };
template <> struct LaneOf<double> { typedef double T; };

__device__ __forceinline__ float2 ladd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 lneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 lsub(float2 a, float2 b) { return __fadd2_rn(a, lneg(b)); }
__device__ __forceinline__ float2 lmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 lfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double ladd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double lneg(double a) { return -a; }
__device__ __forceinline__ double lsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double lmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double lfma(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename L> __device__ __forceinline__ L lbc(double v);
template <> __device__ __forceinline__ float2 lbc<float2>(double v) { return make_float2((float)v, (float)v); }
template <> __device__ __forceinline__ double lbc<double>(double v) { return v; }

// The scale of a sum that goes on over further terms of modulus m (ratio: what
// the terms so far are to be multiplied by, an exact power of two).
template <typename L> struct RunScale;
template <> struct RunScale<double> {
  static constexpr double scale = 1.0, inv = 1.0;
  template <typename F> __device__ __forceinline__ void grow(float, F&&) {}
};
template <> struct RunScale<float2> {
  float top = 0.f;
  float2 scale = {1.f, 1.f};
  double inv = 1.0;
  template <typename F> __device__ __forceinline__ void grow(float m, F&& ratio);
};

template <typename L, typename Real> __device__ __forceinline__ L lane_bc(Real v) {
  if constexpr (sizeof(L) == sizeof(Real)) return v;
  else return L{v, v};
}

template <typename L> struct Vec {
  L re, im;
};

template <typename L> __device__ __forceinline__ Vec<L> vadd(const Vec<L>& a, const Vec<L>& b) {
  return {ladd(a.re, b.re), ladd(a.im, b.im)};
}
template <typename L> __device__ __forceinline__ Vec<L> vsub(const Vec<L>& a, const Vec<L>& b) {
  return {lsub(a.re, b.re), lsub(a.im, b.im)};
}
// a + (DIR i) t and a - (DIR i) t
template <int DIR, typename L> __device__ __forceinline__ Vec<L> vadd_i(const Vec<L>& a, const Vec<L>& t) {
  return DIR < 0 ? Vec<L>{ladd(a.re, t.im), lsub(a.im, t.re)} : Vec<L>{lsub(a.re, t.im), ladd(a.im, t.re)};
}
template <int DIR, typename L> __device__ __forceinline__ Vec<L> vsub_i(const Vec<L>& a, const Vec<L>& t) {
  return DIR < 0 ? Vec<L>{lsub(a.re, t.im), ladd(a.im, t.re)} : Vec<L>{ladd(a.re, t.im), lsub(a.im, t.re)};
}
// ---------------------------------------------------------------------------
// float64 sums over float fields. A float64 warp instruction, a conversion
// included, holds its scheduler for 63 cycles, a float one for one or two: the
// products are split exactly (fma) and added up as unevaluated sums of three
// floats (Knuth's two-sum), good to 2^-70 of the sum of moduli, closer than the
// float64 additions they replace; one conversion per thread follows. Observables
// of 128^3: moments 56 -> 33 us, field energy 36.6 -> 17.0, L_z along y 39.6 ->
// 14.1 and along x 38.5 -> 15.9, kinetic energy 28.1 -> 18.7. The terms are scaled by powers
// of two (pow2_scale), so that neither tiny nor large fields lose products to
// the float range. The double version is the plain sum.
// ---------------------------------------------------------------------------
template <typename L> struct ExactSum;
template <> struct ExactSum<float2> {
  float2 s = {0.f, 0.f}, e = {0.f, 0.f}, f = {0.f, 0.f};
  static __device__ __forceinline__ void two_sum(float2 a, float2 b, float2& sum, float2& err) {
    const float2 t = ladd(a, b), bb = lsub(t, a);
    err = ladd(lsub(a, lsub(t, bb)), lsub(b, bb));
    sum = t;
  }
  __device__ __forceinline__ void low(float2 x) {
    float2 t;
    two_sum(e, x, e, t);
    f = ladd(f, t);
  }
  __device__ __forceinline__ void add(float2 x) {
    float2 t;
    two_sum(s, x, s, t);
    low(t);
  }
  __device__ __forceinline__ void prod(float2 a, float2 b) {
    const float2 p = lmul(a, b);
    add(p);
    low(lfma(a, b, lneg(p)));
  }
  __device__ __forceinline__ void add(const ExactSum& x) {
    add(x.s);
    low(x.e);
    f = ladd(f, x.f);
  }
  __device__ __forceinline__ void prod(float2 w, const ExactSum& x) {
    prod(w, x.s);
    const float2 m = lmul(w, x.e);
    low(m);
    f = ladd(f, lfma(w, x.f, lfma(w, x.e, lneg(m))));
  }
  __device__ __forceinline__ void square(const ExactSum& x) {
    const float2 d = ladd(x.s, x.s), m = lmul(d, x.e);
    prod(x.s, x.s);
    low(m);
    f = ladd(f, lfma(d, x.f, lfma(x.e, x.e, lfma(d, x.e, lneg(m)))));
  }
  // re^2 + im^2
  static __device__ __forceinline__ ExactSum density(float2 re, float2 im) {
    ExactSum r;
    const float2 p = lmul(re, re), q = lmul(im, im);
    float2 t, u, v;
    two_sum(p, q, r.s, t);
    two_sum(lfma(re, re, lneg(p)), lfma(im, im, lneg(q)), u, v);
    two_sum(t, u, r.e, t);
    r.f = ladd(t, v);
    return r;
  }
  // w (re^2 + im^2)
  __device__ __forceinline__ void dens(float2 w, float2 re, float2 im) { prod(w, density(re, im)); }
  __device__ __forceinline__ void rescale(float2 w) {
    s = lmul(s, w);
    e = lmul(e, w);
    f = lmul(f, w);
  }
  // an overflow or an infinity leaves the leading sum as it is and the others NaN
  __device__ __forceinline__ double get(int q) const {
    const float a = q ? s.y : s.x, b = q ? e.y : e.x, c = q ? f.y : f.x;
    return isfinite(a) ? (double)a + ((double)b + (double)c) : (double)a;
  }
};
template <> struct ExactSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ void prod(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ void dens(double w, double re, double im) { s += w * (re * re + im * im); }
  __device__ __forceinline__ void rescale(double) {}
  __device__ __forceinline__ double get(int) const { return s; }
};

// max of m and the lanes' moduli (unused for double)
__device__ __forceinline__ float lmax_abs(float m, float2 v) { return fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))); }
__device__ __forceinline__ float lmax_abs(float m, double) { return m; }
// The power of two that takes m near 1, and its inverse; 1 for zero, infinity and NaN.
template <typename L> struct Pow2 {
  L scale;
  double inv;
};
template <typename L> __device__ __forceinline__ Pow2<L> pow2_scale(float m);
template <> __device__ __forceinline__ Pow2<double> pow2_scale<double>(float) { return {1.0, 1.0}; }
template <> __device__ __forceinline__ Pow2<float2> pow2_scale<float2>(float m) {
  int e = (__float_as_int(m) >> 23) & 255;
  if (e == 255 || m == 0.f) e = 127;
  e = min(max(e, 1), 253);
  const float s = __int_as_float((254 - e) << 23);
  return {make_float2(s, s), (double)__int_as_float(e << 23)};
}

template <typename F> __device__ __forceinline__ void RunScale<float2>::grow(float m, F&& ratio) {
  if (!(m > top)) return;
  const Pow2<float2> p = pow2_scale<float2>(m);
  if (top > 0.f) {
    const float r = p.scale.x * (float)inv;
    ratio(make_float2(r, r));
  }
  top = m;
  scale = p.scale;
  inv = p.inv;
}

// head and tail of a constant in the lane's precision (folded at compile time)
__device__ __forceinline__ void head_tail(double k, float2& h, float2& t) {
  h = make_float2((float)k, (float)k);
  const float r = (float)(k - (double)(float)k);
  t = make_float2(r, r);
}
__device__ __forceinline__ void head_tail(double k, double& h, double& t) {
  h = k;
  t = 0.0;
}
template <bool EXACT, typename L> struct TwoTerm { static constexpr bool v = false; };
template <> struct TwoTerm<true, float2> { static constexpr bool v = true; };

// x times an irrational constant, rounded once (float: head and tail, in every
// transform: sqrt(1/2) and sqrt(3)/2 are 1.7e-8 off as floats, and that gain
// on half of the modes is what the dipolar energy, a small difference of large
// ones, sees of a density transform's errors)
template <bool EXACT, typename L> __device__ __forceinline__ L lkmul(L x, double k) {
  L h, t;
  head_tail(k, h, t);
  if constexpr (TwoTerm<true, L>::v) return lfma(x, h, lmul(x, t));
  else return lmul(x, h);
}
// a times the constant c + i DIR s, head and tail likewise: the plain rounded
// pairs are 2.9e-8 (16th roots) and 1.3e-8 (12th) short, and a zero-padded pass
// has them on its odd outputs alone (field energy of 128^3 against 64 bits:
// 5.3e-7 with the heads alone, 9e-8; 128^3 step 441 -> 445 us for four)
template <int DIR, bool EXACT, typename L> __device__ __forceinline__ Vec<L> vkmul(const Vec<L>& a, double c, double s) {
  L ch, ct, sh, st;
  head_tail(c, ch, ct);
  head_tail(DIR * s, sh, st);
  if constexpr (TwoTerm<true, L>::v)
    return {lfma(a.re, ch, lfma(a.im, lneg(sh), lfma(a.re, ct, lmul(a.im, lneg(st))))),
            lfma(a.re, sh, lfma(a.im, ch, lfma(a.re, st, lmul(a.im, ct))))};
  else
    return {lfma(a.re, ch, lmul(a.im, lneg(sh))), lfma(a.re, sh, lmul(a.im, ch))};
}
// a times exp(DIR i pi / 4) (ODD false) or exp(DIR 3 i pi / 4) (ODD true)
template <int DIR, bool EXACT, bool ODD, typename L> __device__ __forceinline__ Vec<L> veighth(const Vec<L>& a) {
  const double h = 0.70710678118654752440084436210484904;
  const Vec<L> t = vadd_i<DIR>(a, a);  // (1 + DIR i) a
  if constexpr (!ODD) return {lkmul<EXACT>(t.re, h), lkmul<EXACT>(t.im, h)};
  // (-1 + DIR i) a = DIR i (1 + DIR i) a
  else if constexpr (DIR < 0) return {lkmul<EXACT>(t.im, h), lkmul<EXACT>(t.re, -h)};
  else return {lkmul<EXACT>(t.im, -h), lkmul<EXACT>(t.re, h)};
}

// ---------------------------------------------------------------------------
// DFTs of 2, 3, 4, 6, 8, 12 and 16 elements in registers, natural order in and out
// ---------------------------------------------------------------------------
template <typename L> __device__ __forceinline__ void vdft2(Vec<L>& a, Vec<L>& b) {
  const Vec<L> t = a;
  a = vadd(t, b);
  b = vsub(t, b);
}
template <int DIR, typename L>
__device__ __forceinline__ void vdft4(Vec<L>& a0, Vec<L>& a1, Vec<L>& a2, Vec<L>& a3) {
  const Vec<L> s02 = vadd(a0, a2), d02 = vsub(a0, a2), s13 = vadd(a1, a3), t13 = vsub(a1, a3);
  a0 = vadd(s02, s13);
  a2 = vsub(s02, s13);
  a1 = vadd_i<DIR>(d02, t13);
  a3 = vsub_i<DIR>(d02, t13);
}
template <int DIR, bool EXACT, typename L>
__device__ __forceinline__ void vdft3(Vec<L>& a0, Vec<L>& a1, Vec<L>& a2) {
  const double s3 = 0.86602540378443864676372317075293618;  // sqrt(3)/2
  const L mh = lbc<L>(-0.5);
  const Vec<L> t = vadd(a1, a2), d = vsub(a1, a2);
  const Vec<L> m{lfma(mh, t.re, a0.re), lfma(mh, t.im, a0.im)};
  const Vec<L> e{lkmul<EXACT>(d.re, s3), lkmul<EXACT>(d.im, s3)};
  a0 = vadd(a0, t);
  a1 = vadd_i<DIR>(m, e);
  a2 = vsub_i<DIR>(m, e);
}
template <int DIR, bool EXACT, typename L> __device__ __forceinline__ void vdft8(Vec<L>* v) {
  vdft4<DIR>(v[0], v[2], v[4], v[6]);
  vdft4<DIR>(v[1], v[3], v[5], v[7]);
  const Vec<L> t1 = veighth<DIR, EXACT, false>(v[3]), o2 = v[5], t3 = veighth<DIR, EXACT, true>(v[7]);
  const Vec<L> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
  v[0] = vadd(e0, o0);
  v[4] = vsub(e0, o0);
  v[1] = vadd(e1, t1);
  v[5] = vsub(e1, t1);
  v[2] = vadd_i<DIR>(e2, o2);
  v[6] = vsub_i<DIR>(e2, o2);
  v[3] = vadd(e3, t3);
  v[7] = vsub(e3, t3);
}
// 16 = 4 x 4: columns b over v[4a + b], twiddles w16^{bc}, rows c, output c + 4d
template <int DIR, bool EXACT, typename L> __device__ __forceinline__ void vdft16(Vec<L>* v) {
  const double c1 = 0.92387953251128675612818318939679, s1 = 0.38268343236508977172845998403040;
#pragma unroll
  for (int b = 0; b < 4; ++b) vdft4<DIR>(v[b], v[4 + b], v[8 + b], v[12 + b]);
  v[5] = vkmul<DIR, EXACT>(v[5], c1, s1);            // w^1
  v[9] = veighth<DIR, EXACT, false>(v[9]);           // w^2
  v[13] = vkmul<DIR, EXACT>(v[13], s1, c1);          // w^3
  v[6] = veighth<DIR, EXACT, false>(v[6]);           // w^2
  v[14] = veighth<DIR, EXACT, true>(v[14]);          // w^6
  v[7] = vkmul<DIR, EXACT>(v[7], s1, c1);            // w^3
  v[11] = veighth<DIR, EXACT, true>(v[11]);          // w^6
  v[15] = vkmul<DIR, EXACT>(v[15], -c1, -s1);        // w^9
  const Vec<L> t10 = v[10];                          // w^4 = DIR i, merged into the row transform below
  vdft4<DIR>(v[0], v[1], v[2], v[3]);
  vdft4<DIR>(v[4], v[5], v[6], v[7]);
  {
    const Vec<L> s02 = vadd_i<DIR>(v[8], t10), d02 = vsub_i<DIR>(v[8], t10), s13 = vadd(v[9], v[11]),
                 t13 = vsub(v[9], v[11]);
    v[8] = vadd(s02, s13);
    v[10] = vsub(s02, s13);
    v[9] = vadd_i<DIR>(d02, t13);
    v[11] = vsub_i<DIR>(d02, t13);
  }
  vdft4<DIR>(v[12], v[13], v[14], v[15]);
  // v[4c + d] holds output c + 4d
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int d = c + 1; d < 4; ++d) {
      const Vec<L> t = v[4 * c + d];
      v[4 * c + d] = v[4 * d + c];
      v[4 * d + c] = t;
    }
}
// 6 = 2 x 3 and 12 = 4 x 3 by the prime-factor index maps (no twiddles)
template <int DIR, bool EXACT, typename L> __device__ __forceinline__ void vdft6(Vec<L>* v) {
  Vec<L> u[2][3];
#pragma unroll
  for (int n1 = 0; n1 < 2; ++n1) {
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) u[n1][n2] = v[(3 * n1 + 2 * n2) % 6];
    vdft3<DIR, EXACT>(u[n1][0], u[n1][1], u[n1][2]);
  }
#pragma unroll
  for (int k2 = 0; k2 < 3; ++k2) {
    vdft2(u[0][k2], u[1][k2]);
#pragma unroll
    for (int k1 = 0; k1 < 2; ++k1) v[(3 * k1 + 4 * k2) % 6] = u[k1][k2];
  }
}
template <int DIR, bool EXACT, typename L> __device__ __forceinline__ void vdft12(Vec<L>* v) {
  Vec<L> u[4][3];
#pragma unroll
  for (int n1 = 0; n1 < 4; ++n1) {
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) u[n1][n2] = v[(3 * n1 + 4 * n2) % 12];
    vdft3<DIR, EXACT>(u[n1][0], u[n1][1], u[n1][2]);
  }
#pragma unroll
  for (int k2 = 0; k2 < 3; ++k2) {
    vdft4<DIR>(u[0][k2], u[1][k2], u[2][k2], u[3][k2]);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) v[(9 * k1 + 4 * k2) % 12] = u[k1][k2];
  }
}
template <int R, int DIR, bool EXACT, typename L> __device__ __forceinline__ void vdft(Vec<L>* v) {
  if constexpr (R == 2) vdft2(v[0], v[1]);
  else if constexpr (R == 3) vdft3<DIR, EXACT>(v[0], v[1], v[2]);
  else if constexpr (R == 4) vdft4<DIR>(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 6) vdft6<DIR, EXACT>(v);
  else if constexpr (R == 8) vdft8<DIR, EXACT>(v);
  else if constexpr (R == 12) vdft12<DIR, EXACT>(v);
  else {
    static_assert(R == 16, "radix");
    vdft16<DIR, EXACT>(v);
  }
}

// The same with the second half of the inputs zero (a zero-padded line; v[R/2..]
// is not read): even outputs are the DFT of size R/2 of the inputs, odd ones
// that of the inputs times w_R^r.
template <int R, int DIR, bool EXACT, typename L> __device__ __forceinline__ void vdft_zh(Vec<L>* v) {
  constexpr int H = R / 2;
  static_assert(R % 2 == 0 && H * 2 == R, "zero-padded passes have an even radix");
  // cos and sin of 2 pi r / R, r < R / 2
  constexpr double h = 0.70710678118654752440084436210484904;
  constexpr double q = 0.86602540378443864676372317075293618;
  constexpr double c12[6] = {1.0, q, 0.5, 0.0, -0.5, -q}, s12[6] = {0.0, 0.5, q, 1.0, q, 0.5};
  constexpr double a = 0.92387953251128675612818318939679, b = 0.38268343236508977172845998403040;
  constexpr double c16[8] = {1.0, a, h, b, 0.0, -b, -h, -a}, s16[8] = {0.0, b, h, a, 1.0, a, h, b};
  Vec<L> o[H];
#pragma unroll
  for (int r = 0; r < H; ++r) {
    if (r == 0) o[r] = v[r];
    else if (4 * r == R) o[r] = DIR < 0 ? Vec<L>{v[r].im, lneg(v[r].re)} : Vec<L>{lneg(v[r].im), v[r].re};
    else if (8 * r == R) o[r] = veighth<DIR, EXACT, false>(v[r]);
    else if (8 * r == 3 * R) o[r] = veighth<DIR, EXACT, true>(v[r]);
    else if (R == 16) o[r] = vkmul<DIR, EXACT>(v[r], c16[r & 7], s16[r & 7]);
    else o[r] = vkmul<DIR, EXACT>(v[r], c12[(12 / R) * r % 6], s12[(12 / R) * r % 6]);
  }
  vdft<H, DIR, EXACT>(v);
  vdft<H, DIR, EXACT>(o);
  Vec<L> e[H];
#pragma unroll
  for (int r = 0; r < H; ++r) e[r] = v[r];
#pragma unroll
  for (int r = 0; r < H; ++r) {
    v[2 * r] = e[r];
    v[2 * r + 1] = o[r];
  }
}

// ---------------------------------------------------------------------------
// twiddles: w = exp(-2 pi i m / L) from a table (conjugated for DIR > 0). Float:
// head (c, c, s, s) at t[0] and remainder at t[tail]; double: (c, s).
// ---------------------------------------------------------------------------
template <int DIR, bool EXACT>
__device__ __forceinline__ Vec<float2> vtwiddle(const Vec<float2>& v, const float4* __restrict__ t, int tail) {
  const float4 w = __ldg(t);
  const float2 c = make_float2(w.x, w.y), s0 = make_float2(w.z, w.w);
  const float2 s = DIR < 0 ? s0 : lneg(s0);
  if constexpr (EXACT) {
    const float4 l = __ldg(t + tail);
    const float2 lc = make_float2(l.x, l.y), l0 = make_float2(l.z, l.w);
    const float2 ls = DIR < 0 ? l0 : lneg(l0);
    return {lfma(v.re, c, lfma(v.im, lneg(s), lfma(v.re, lc, lmul(v.im, lneg(ls))))),
            lfma(v.re, s, lfma(v.im, c, lfma(v.re, ls, lmul(v.im, lc))))};
  } else {
    return {lfma(v.re, c, lmul(v.im, lneg(s))), lfma(v.re, s, lmul(v.im, c))};
  }
}
template <int DIR, bool EXACT>
__device__ __forceinline__ Vec<double> vtwiddle(const Vec<double>& v, const double2* __restrict__ t, int) {
  const double2 w = __ldg(t);
  const double c = w.x, s = DIR < 0 ? w.y : -w.y;
  return {lfma(v.re, c, lmul(v.im, -s)), lfma(v.re, s, lmul(v.im, c))};
}

// a + w b and a - w b for w = c (1 + i t), t negated for DIR > 0 by the caller
__device__ __forceinline__ void tan_bfly(Vec<double>& a, Vec<double>& b, double c, double t) {
  const double ur = lfma(b.im, -t, b.re), ui = lfma(b.re, t, b.im);
  b = {lfma(-c, ur, a.re), lfma(-c, ui, a.im)};
  a = {lfma(c, ur, a.re), lfma(c, ui, a.im)};
}
// the same with DIR i w
template <int DIR> __device__ __forceinline__ void tan_bfly_i(Vec<double>& a, Vec<double>& b, double c, double t) {
  const double ur = lfma(b.im, -t, b.re), ui = lfma(b.re, t, b.im), d = DIR * c;
  b = {lfma(d, ui, a.re), lfma(-d, ur, a.im)};
  a = {lfma(-d, ui, a.re), lfma(d, ur, a.im)};
}
// Twiddled butterflies of radix 2 and 4 (inputs not multiplied yet), natural order
template <int DIR> __device__ __forceinline__ void tan_dft2(Vec<double>* v, const double2* __restrict__ t, int ns) {
  const double2 w = __ldg(t + ns);
  tan_bfly(v[0], v[1], w.x, DIR < 0 ? w.y : -w.y);
}
template <int DIR> __device__ __forceinline__ void tan_dft4(Vec<double>* v, const double2* __restrict__ t, int ns) {
  const double2 w1 = __ldg(t + ns), w2 = __ldg(t + 2 * ns);
  const double t1 = DIR < 0 ? w1.y : -w1.y, t2 = DIR < 0 ? w2.y : -w2.y;
  Vec<double> s02 = v[0], d02 = v[2], s13 = v[1], d13 = v[3];
  tan_bfly(s02, d02, w2.x, t2);         // a0 +- w^2 a2
  tan_bfly(s13, d13, w2.x, t2);         // a1 +- w^2 a3
  tan_bfly(s02, s13, w1.x, t1);         // outputs 0 and 2
  tan_bfly_i<DIR>(d02, d13, w1.x, t1);  // outputs 1 and 3
  v[0] = s02;
  v[1] = d02;
  v[2] = s13;
  v[3] = d13;
}

// 16-byte slot of an exchange tile
template <typename L> __device__ __forceinline__ void slot_st(float4* buf, int s, const Vec<L>& v);
template <> __device__ __forceinline__ void slot_st(float4* buf, int s, const Vec<float2>& v) {
  buf[s] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
}
template <> __device__ __forceinline__ void slot_st(float4* buf, int s, const Vec<double>& v) {
  reinterpret_cast<double2*>(buf)[s] = make_double2(v.re, v.im);
}
__device__ __forceinline__ void slot_ld(const float4* buf, int s, Vec<float2>& v) {
  const float4 t = buf[s];
  v = {make_float2(t.x, t.y), make_float2(t.z, t.w)};
}
__device__ __forceinline__ void slot_ld(const float4* buf, int s, Vec<double>& v) {
  const double2 t = reinterpret_cast<const double2*>(buf)[s];
  v = {t.x, t.y};
}

// ---------------------------------------------------------------------------
// plans: radices, and threads per transform (T). Pass p has N / R_p items, item
// j of it reading positions j + r N/R_p; thread it of a transform takes items
// it, it + T, ... (some threads are idle in a pass with fewer items than T).
// ---------------------------------------------------------------------------
struct FftPlan {
  int np, r[4], T;
};
// Float plans: the fewest passes that fit 16 elements (64 registers) per thread.
// Double plans: radices up to 8 and four elements per thread in most passes:
// a float64 warp instruction holds its scheduler for 64 cycles (two lanes per
// cycle and SM), so the operations are what counts, not the exchanges, and
// many threads with short chains fill a small grid's SMs. Every pass keeps whole
// warps busy: idle lanes cost as much as active ones.
__host__ __device__ constexpr FftPlan fft_plan(int n, bool f64) {
  if (f64) switch (n) {
      case 8: return {2, {4, 2, 1, 1}, 2};
      case 12: return {2, {4, 3, 1, 1}, 4};
      case 16: return {2, {4, 4, 1, 1}, 4};
      case 24: return {2, {4, 6, 1, 1}, 6};
      case 32: return {3, {4, 4, 2, 1}, 8};
      case 48: return {3, {4, 3, 4, 1}, 12};
      case 64: return {3, {4, 4, 4, 1}, 16};
      case 96: return {3, {4, 6, 4, 1}, 24};
      case 128: return {4, {4, 4, 2, 4}, 32};
      case 192: return {4, {4, 4, 3, 4}, 48};
      case 256: return {4, {4, 4, 4, 4}, 64};
      case 384: return {4, {4, 4, 6, 4}, 96};
      case 512: return {4, {4, 8, 4, 4}, 128};
      case 768: return {4, {4, 8, 6, 4}, 192};
      default: return {4, {4, 8, 8, 4}, 256};
    }
  switch (n) {
    case 16: return {2, {4, 4, 1, 1}, 4};
    case 24: return {2, {6, 4, 1, 1}, 6};
    case 32: return {2, {8, 4, 1, 1}, 4};
    case 48: return {2, {8, 6, 1, 1}, 8};
    case 64: return {2, {8, 8, 1, 1}, 8};
    case 96: return {2, {12, 8, 1, 1}, 12};
    case 128: return {2, {16, 8, 1, 1}, 8};
    case 192: return {2, {16, 12, 1, 1}, 16};
    case 256: return {2, {16, 16, 1, 1}, 16};
    case 384: return {3, {8, 6, 8, 1}, 64};
    case 512: return {3, {8, 8, 8, 1}, 64};
    case 768: return {3, {8, 12, 8, 1}, 64};
    case 1024: return {3, {16, 8, 8, 1}, 64};
    default: return {2, {4, 2, 1, 1}, 2};  // 8 and 12 are only run slim
  }
}

// Float plans of at most eight elements per thread (64 registers) and more
// threads; four elements up to length 64, where a transform is a chain of latencies.
__host__ __device__ constexpr FftPlan fft_plan_slim(int n) {
  switch (n) {
    case 8: return {2, {4, 2, 1, 1}, 2};
    case 12: return {2, {3, 4, 1, 1}, 4};
    case 24: return {2, {4, 6, 1, 1}, 6};
    case 32: return {3, {4, 2, 4, 1}, 8};
    case 48: return {3, {4, 3, 4, 1}, 12};
    case 64: return {3, {4, 4, 4, 1}, 16};
    case 96: return {3, {4, 6, 4, 1}, 16};
    case 128: return {3, {8, 4, 4, 1}, 16};
    case 192: return {3, {8, 6, 4, 1}, 32};
    case 256: return {3, {8, 8, 4, 1}, 32};
    case 768: return {4, {8, 6, 4, 4}, 128};
    case 1024: return {4, {8, 8, 4, 4}, 128};
    default: return fft_plan(n, false);
  }
}

// Float64 passes of radix 2 and 4 take their twiddles as (cos, tan): a product
// with w = c (1 + i t) is only ever added to and subtracted from another
// element, so a +- w b needs two fused operations for u = (1 + i t) b and four
// for a +- c u, six where the product and the sums take eight; a radix-4
// butterfly (w^2 b factored the same way, w^3 = w w^2 by factoring w out of
// the odd pair) takes 24 operations and two twiddles in place of 28 and three.
// On GB300 float64 operations are the whole time of a float64 pass (128^3: one
// transform along y 90 -> 71 us; a step 2.83 -> 2.31 ms).
__host__ __device__ constexpr bool tw_tan(int radix, bool f64) { return f64 && (radix == 2 || radix == 4); }

// Twiddle tables of a transform length: one per plan (large radices, slim) and
// radix order (as listed, reversed), each listing pass after pass (the first
// has no twiddles) the factors exp(-2 pi i k r / (NS R)) as [r][k], r < R,
// k < NS: the threads of a warp, whose items k are neighbours, read
// neighbouring entries, at a constant distance for every r. (With one table
// per length, entry k r N / (NS R), the 16 lines of a warp's entries made the
// 256^3 x transform 55 us; this order 42.) A table holds at
// most 3N/2 entries; float ones are followed by their remainders.
__host__ __device__ constexpr int tw_entries(int n) { return 3 * n / 2; }
__host__ __device__ constexpr int tw_tables(bool f64) { return f64 ? 2 : 4; }
// bytes of the tables of length n: (c, c, s, s) heads and tails, or (c, s)
__host__ __device__ constexpr size_t tw_bytes(int n, bool f64) {
  return (size_t)tw_tables(f64) * tw_entries(n) * (f64 ? 16 : 32);
}

template <typename Real> struct TwOf;
template <> struct TwOf<float> { typedef float4 T; };
template <> struct TwOf<double> { typedef double2 T; };

// Reads a range of a constant table into L1 (the values go to `sink`, a shared
// word per thread that is overwritten before it is read).
__device__ __forceinline__ unsigned warm_line(const void* p) { return __ldg(reinterpret_cast<const unsigned*>(p)); }
template <int BYTES, int NT> __device__ __forceinline__ unsigned warm(const void* p, int tid) {
  constexpr int I = (BYTES + 128 * NT - 1) / (128 * NT);
  unsigned x[I], s = 0;
#pragma unroll
  for (int i = 0; i < I; ++i) {
    const int o = (tid + i * NT) * 128;
    x[i] = o < BYTES ? warm_line(static_cast<const char*>(p) + o) : 0u;
  }
#pragma unroll
  for (int i = 0; i < I; ++i) s ^= x[i];
  return s;
}

// Transform of length N by TT threads (0: the plan's T).
template <typename Real, int N, int TT = 0, bool SLIM = false>
struct FftCfg {
  typedef typename LaneOf<Real>::T L;
  static constexpr bool F64 = sizeof(Real) == 8;
  typedef typename TwOf<Real>::T W;  // a twiddle table entry
  static constexpr FftPlan P = SLIM && sizeof(Real) == 4 ? fft_plan_slim(N) : fft_plan(N, sizeof(Real) == 8);
  static constexpr int T = TT ? TT : P.T;
  // radix and items per thread of pass p, taken in reverse order when REV
  __host__ __device__ static constexpr int R(int p, bool rev) { return P.r[rev ? P.np - 1 - p : p]; }
  __host__ __device__ static constexpr int I(int p, bool rev) { return (N / R(p, rev) + T - 1) / T; }
  __host__ __device__ static constexpr int elems() {
    int e = 0;
    for (int p = 0; p < P.np; ++p) {
      const int v = R(p, false) * I(p, false);
      e = v > e ? v : e;
    }
    return e;
  }
  static constexpr int E = elems();  // elements a thread holds
  static constexpr int RF = P.r[0], RL = P.r[P.np - 1];

  // whether item i of thread `it` exists in a pass of radix RX
  template <int RX> __device__ __forceinline__ static bool ok(int it, int i) {
    return (N / RX) % T == 0 || it + i * T < N / RX;
  }
  // the elements of a pass of radix RX: f(register index, position, r), positions j + r N/RX
  template <int RX, typename F> __device__ __forceinline__ static void each(int it, F&& f) {
#pragma unroll
    for (int i = 0; i < (N / RX + T - 1) / T; ++i) {
      if (!ok<RX>(it, i)) continue;
      const int j = it + i * T;
#pragma unroll
      for (int r = 0; r < RX; ++r) f(i * RX + r, j + r * (N / RX), r);
    }
  }

  // first entry of pass p in the plan's table, and the table's place
  __host__ __device__ static constexpr int tw_off(int p, bool rev) {
    int off = ((!F64 && SLIM ? 2 : 0) + (rev ? 1 : 0)) * (F64 ? 1 : 2) * tw_entries(N), ns = R(0, rev);
    for (int q = 1; q < p; ++q) {
      ns *= R(q, rev);
      off += ns;
    }
    return off;
  }

  // entries of the plan's table in one radix order
  __host__ __device__ static constexpr int tw_count(bool rev) {
    int n = 0, ns = R(0, rev);
    for (int q = 1; q < P.np; ++q) {
      ns *= R(q, rev);
      n += ns;
    }
    return n;
  }
  // that table into L1
  template <bool REV, bool EXACT, int NT> __device__ __forceinline__ static unsigned warm_table(const W* tw, int tid) {
    constexpr int off = tw_off(1, REV), n = tw_count(REV) * (int)sizeof(W);
    unsigned x = warm<n, NT>(tw + off, tid);
    if constexpr (!F64 && EXACT) x ^= warm<n, NT>(tw + off + tw_entries(N), tid);
    return x;
  }

  // One pass on the registers: twiddles (NS > 1, this pass's table at tw) and the radix-RX DFTs.
  template <int DIR, bool EXACT, int RX, int NS, bool ZIN>
  __device__ __forceinline__ static void pass(Vec<L> (&v)[E], const W* __restrict__ tw, int it) {
#pragma unroll
    for (int i = 0; i < (N / RX + T - 1) / T; ++i) {
      if (!ok<RX>(it, i)) continue;
      if constexpr (NS > 1 && tw_tan(RX, F64)) {
        const W* __restrict__ t = tw + (it + i * T) % NS;
        if constexpr (RX == 2) tan_dft2<DIR>(&v[i * RX], t, NS);
        else tan_dft4<DIR>(&v[i * RX], t, NS);
        continue;
      } else if constexpr (NS > 1) {
        const W* __restrict__ t = tw + (it + i * T) % NS;
#pragma unroll
        for (int r = 1; r < RX; ++r) v[i * RX + r] = vtwiddle<DIR, EXACT>(v[i * RX + r], t + r * NS, tw_entries(N));
      }
      if constexpr (ZIN) vdft_zh<RX, DIR, EXACT>(&v[i * RX]);
      else vdft<RX, DIR, EXACT>(&v[i * RX]);
    }
  }

  // Passes PASS..last of the transform whose first inputs are in v. A: the
  // tile's address map, slot(row) for this thread's column or line
  // (A::slot<FR>(row), FR the first radix: rows written by the first pass lie
  // FR apart). Every exchange is store, barrier, load; the barrier that frees
  // the tile for the next store comes right before that store (DIRTY: the tile
  // may still be read by other threads when the first exchange stores), so
  // that warps drift apart over a whole pass. Ends with the tile possibly
  // still being read. ZIN: positions >= N/2 of the input are zero (not read).
  template <int DIR, bool EXACT, bool REV, bool DIRTY, bool ZIN = false, int PASS = 0, int NS = 1, typename A>
  __device__ __forceinline__ static void run(Vec<L> (&v)[E], float4* buf, const A& addr, const W* __restrict__ tw, int it) {
    constexpr int RX = R(PASS, REV), FR = R(0, REV);
    pass<DIR, EXACT, RX, NS, ZIN && PASS == 0>(v, tw + tw_off(PASS, REV), it);
    if constexpr (PASS + 1 < P.np) {
      constexpr int R2 = R(PASS + 1, REV);
      if constexpr (DIRTY || PASS > 0) addr.sync();
#pragma unroll
      for (int i = 0; i < (N / RX + T - 1) / T; ++i) {
        if (!ok<RX>(it, i)) continue;
        const int j = it + i * T, base = (j / NS) * NS * RX + j % NS;
#pragma unroll
        for (int r = 0; r < RX; ++r) slot_st(buf, addr.template slot<FR>(base + r * NS), v[i * RX + r]);
      }
      addr.sync();
      each<R2>(it, [&](int e, int row, int) { slot_ld(buf, addr.template slot<FR>(row), v[e]); });
      run<DIR, EXACT, REV, DIRTY, ZIN, PASS + 1, NS * RX>(v, buf, addr, tw, it);
    }
  }
};

}  // namespace fse
