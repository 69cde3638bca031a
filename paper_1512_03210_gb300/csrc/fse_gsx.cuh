// fse_gsx.cuh -- the x passes of the ground-state operator, with the Krylov vector work fused in.
//
// One product of the preconditioned operator, (I + P_Delta A_TF) u, is
//   gs_fwd   u (formed on the fly from the BiCGStab vectors), A_TF u = W u -
//            Omega L_z u, forward transform along x
//   the passes along y (and z) with P_Delta in between (COL_RMUL)
//   gs_inv   inverse transform along x, u + P_Delta A_TF u, and the partial
//            inner products that the next scalar needs
// so that a product in 2D is three launches (512^2 float64: an iteration of two
// products went from 40 launches and 0.43 ms to 10), and no vector is read
// for its update alone.
#pragma once

#include "fse_launch.cuh"

namespace fse {

// BiCGStab scalars on the device (see fse_ground.cu)
enum { SC_RHO = 0, SC_RHOP = 2, SC_ALPHA = 4, SC_OM = 6, SC_BETA = 8, SC_BN = 10, SC_RES = 11, SC_DONE = 12,
       SC_IT = 13, SC_TOL = 14, SC_SIZE = 16 };

// u of a product: U_PLAIN a; U_P a + beta (o - omega c) (a on the first
// iteration), written back to o; U_S a - alpha c, written to o. With the solve
// done, o stays as it is.
enum { U_PLAIN = 0, U_P = 1, U_S = 2 };
struct GsFwd {
  int mode, nlines, ny;
  const void *a, *c;
  void* o;
  const void* W;        // real field; null: A_TF u = scale u
  double scale;
  const void* dy;       // d_y u (null: no rotation)
  double omega, lo0, h0, lo1, h1, dkx;
  const double* sc;
  void* out;            // x-spectrum of A_TF u
};

// Results of the inverse: V_ADD y = u + d, partials of <rh, y>; V_ADD2 the same
// with <y, u>, <y, y>; V_SET y = d; V_RES y = b - (u + d), copied to y2, with
// <b, b>, <y, y>.
enum { V_ADD = 0, V_ADD2 = 1, V_SET = 2, V_RES = 3 };
struct GsInv {
  int mode, nlines;
  const void *in, *u, *q;  // q: rh (V_ADD) or b (V_RES)
  void *y, *y2;
  double* part;            // 4 values per tile, `stride` partials apart
  int stride;
};

__device__ __forceinline__ double2 gs_ld2(const double* p) { return make_double2(p[0], p[1]); }
__device__ __forceinline__ double2 gs_mul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a + (cx + i cy) b
template <typename L> __device__ __forceinline__ Vec<L> vaxpy(const Vec<L>& a, L cx, L cy, const Vec<L>& b) {
  return {lfma(cx, b.re, lfma(lneg(cy), b.im, a.re)), lfma(cx, b.im, lfma(cy, b.re, a.im))};
}
// sum over the lanes of conj(a) b in float64
__device__ __forceinline__ void dot_add(const Vec<double>& a, const Vec<double>& b, double& re, double& im) {
  re = lfma(a.re, b.re, lfma(a.im, b.im, re));
  im = lfma(a.re, b.im, lfma(-a.im, b.re, im));
}
__device__ __forceinline__ void dot_add(const Vec<float2>& a, const Vec<float2>& b, double& re, double& im) {
  dot_add(Vec<double>{(double)a.re.x, (double)a.im.x}, Vec<double>{(double)b.re.x, (double)b.im.x}, re, im);
  dot_add(Vec<double>{(double)a.re.y, (double)a.im.y}, Vec<double>{(double)b.re.y, (double)b.im.y}, re, im);
}
__device__ __forceinline__ void norm_add(const Vec<double>& a, double& re) { re = lfma(a.re, a.re, lfma(a.im, a.im, re)); }
__device__ __forceinline__ void norm_add(const Vec<float2>& a, double& re) {
  norm_add(Vec<double>{(double)a.re.x, (double)a.im.x}, re);
  norm_add(Vec<double>{(double)a.re.y, (double)a.im.y}, re);
}

// Real values of a group's lines (exist: nl lines from line0 on).
template <int NX> __device__ __forceinline__ float2 rline_ld(const float* line0, int g, int nl, int x) {
  return make_float2(2 * g < nl ? line0[(2 * g) * NX + x] : 0.f, 2 * g + 1 < nl ? line0[(2 * g + 1) * NX + x] : 0.f);
}
template <int NX> __device__ __forceinline__ double rline_ld(const double* line0, int g, int nl, int x) {
  return g < nl ? line0[g * NX + x] : 0.0;
}

template <typename Real, int NX, int LN, bool ROT>
__global__ void __launch_bounds__(XCfg<Real, NX, LN>::NT, XCfg<Real, NX, LN>::minb())
k_gs_fwd(GsFwd a, const typename TwOf<Real>::T* __restrict__ twn) {
  typedef XCfg<Real, NX, LN> K;
  typedef typename K::F1 F1;
  typedef typename K::L L;
  typedef typename Cplx<Real>::T C;
  constexpr int CW = K::CW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* buf = reinterpret_cast<float4*>(smem_raw);
  const int tid = threadIdx.x;
  int it = tid % K::T;
  const int g = tid / K::T, l0 = blockIdx.x * LN, nl = a.nlines - l0;
  const XAddr ad{g * K::LS1};
  pass_prologue();
  const long long off = (long long)l0 * NX;
  Vec<L> v[F1::E], ud[ROT ? F1::E : 1];
  const bool done = a.mode != U_PLAIN && a.sc[SC_DONE] != 0.0;
  if (a.mode == U_PLAIN || done) {
    const C* src = reinterpret_cast<const C*>(done ? a.o : a.a) + off;
    F1::template each<F1::RF>(it, [&](int e, int x, int) { v[e] = line_ld<NX>(src, g, nl, x); });
  } else {
    const C *pa = reinterpret_cast<const C*>(a.a) + off, *pc = reinterpret_cast<const C*>(a.c) + off;
    C* po = reinterpret_cast<C*>(a.o) + off;
    const double2 al = gs_ld2(a.sc + SC_ALPHA), om = gs_ld2(a.sc + SC_OM), be = gs_ld2(a.sc + SC_BETA);
    if (a.mode == U_S) {
      const L cx = lbc<L>(-al.x), cy = lbc<L>(-al.y);
      F1::template each<F1::RF>(it, [&](int e, int x, int) {
        v[e] = vaxpy(line_ld<NX>(pa, g, nl, x), cx, cy, line_ld<NX>(pc, g, nl, x));
        line_st<NX>(po, g, nl, x, v[e]);
      });
    } else if (a.sc[SC_IT] == 0.0) {
      F1::template each<F1::RF>(it, [&](int e, int x, int) {
        v[e] = line_ld<NX>(pa, g, nl, x);
        line_st<NX>(po, g, nl, x, v[e]);
      });
    } else {
      const double2 bo = gs_mul(be, om);
      const L bx = lbc<L>(be.x), by = lbc<L>(be.y), cx = lbc<L>(-bo.x), cy = lbc<L>(-bo.y);
      F1::template each<F1::RF>(it, [&](int e, int x, int) {
        const Vec<L> p = line_ld<NX>((const C*)po, g, nl, x);
        v[e] = vaxpy(vaxpy(line_ld<NX>(pa, g, nl, x), cx, cy, line_ld<NX>(pc, g, nl, x)), bx, by, p);
        line_st<NX>(po, g, nl, x, v[e]);
      });
    }
  }
  if constexpr (ROT) {
    // -Omega L_z u = i Omega (x d_y u - y d_x u), d_x by the lines' own transforms
#pragma unroll
    for (int e = 0; e < F1::E; ++e) ud[e] = v[e];
    F1::template run<-1, true, false, false>(v, buf, ad, twn, it);
    const L inv = lbc<L>(a.dkx / NX);
    F1::template each<F1::RL>(it, [&](int e, int k, int) {
      // i k, the odd factor zero at the Nyquist index
      const L kk = lmul(inv, lbc<L>(2 * k == NX ? Real(0) : Real(wrap_index(k, NX))));
      v[e] = {lneg(lmul(kk, v[e].im)), lmul(kk, v[e].re)};
    });
    F1::template run<+1, true, true, true>(v, buf, ad, twn, it);
    const C* dy = reinterpret_cast<const C*>(a.dy) + off;
    Real yl[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q) yl[q] = Real(-a.omega * (a.lo1 + a.h1 * ((l0 + CW * g + q) % a.ny)));
    const L my = lane_of(yl);
    F1::template each<F1::RF>(it, [&](int e, int x, int) {
      const L ox = lbc<L>(a.omega * (a.lo0 + a.h0 * x));
      const Vec<L> d = line_ld<NX>(dy, g, nl, x);
      // i (ox d + my v)
      const L re = lfma(ox, d.re, lmul(my, v[e].re)), im = lfma(ox, d.im, lmul(my, v[e].im));
      const L w = a.W ? rline_ld<NX>(reinterpret_cast<const Real*>(a.W) + off, g, nl, x) : lbc<L>(a.scale);
      v[e] = {lfma(w, ud[e].re, lneg(im)), lfma(w, ud[e].im, re)};
    });
    F1::template run<-1, true, false, true>(v, buf, ad, twn, it);
  } else {
    F1::template each<F1::RF>(it, [&](int e, int x, int) {
      const L w = a.W ? rline_ld<NX>(reinterpret_cast<const Real*>(a.W) + off, g, nl, x) : lbc<L>(a.scale);
      v[e] = {lmul(w, v[e].re), lmul(w, v[e].im)};
    });
    F1::template run<-1, true, false, false>(v, buf, ad, twn, it);
  }
  C* out = reinterpret_cast<C*>(a.out) + off;
  F1::template each<F1::RL>(it, [&](int e, int x, int) { line_st<NX>(out, g, nl, x, v[e]); });
}

template <typename Real, int NX, int LN>
__global__ void __launch_bounds__(XCfg<Real, NX, LN>::NT, XCfg<Real, NX, LN>::minb())
k_gs_inv(GsInv a, const typename TwOf<Real>::T* __restrict__ twn) {
  typedef XCfg<Real, NX, LN> K;
  typedef typename K::F1 F1;
  typedef typename K::L L;
  typedef typename Cplx<Real>::T C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* buf = reinterpret_cast<float4*>(smem_raw);
  const int tid = threadIdx.x;
  int it = tid % K::T;
  const int g = tid / K::T, l0 = blockIdx.x * LN, nl = a.nlines - l0;
  const XAddr ad{g * K::LS1};
  pass_prologue();
  const long long off = (long long)l0 * NX;
  Vec<L> v[F1::E];
  const C* in = reinterpret_cast<const C*>(a.in) + off;
  F1::template each<F1::RF>(it, [&](int e, int x, int) { v[e] = line_ld<NX>(in, g, nl, x); });
  F1::template run<+1, true, false, false>(v, buf, ad, twn, it);
  C* y = reinterpret_cast<C*>(a.y) + off;
  const C *u = reinterpret_cast<const C*>(a.u) + off, *q = reinterpret_cast<const C*>(a.q) + off;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (a.mode == V_SET) {
    F1::template each<F1::RL>(it, [&](int e, int x, int) { line_st<NX>(y, g, nl, x, v[e]); });
    return;
  }
  if (a.mode == V_ADD) {
    F1::template each<F1::RL>(it, [&](int e, int x, int) {
      v[e] = vadd(v[e], line_ld<NX>(u, g, nl, x));
      line_st<NX>(y, g, nl, x, v[e]);
      dot_add(line_ld<NX>(q, g, nl, x), v[e], s[0], s[1]);
    });
  } else if (a.mode == V_ADD2) {
    F1::template each<F1::RL>(it, [&](int e, int x, int) {
      const Vec<L> uu = line_ld<NX>(u, g, nl, x);
      v[e] = vadd(v[e], uu);
      line_st<NX>(y, g, nl, x, v[e]);
      dot_add(v[e], uu, s[0], s[1]);
      norm_add(v[e], s[2]);
    });
  } else {
    C* y2 = reinterpret_cast<C*>(a.y2) + off;
    F1::template each<F1::RL>(it, [&](int e, int x, int) {
      const Vec<L> b = line_ld<NX>(q, g, nl, x);
      v[e] = vsub(b, vadd(v[e], line_ld<NX>(u, g, nl, x)));
      line_st<NX>(y, g, nl, x, v[e]);
      line_st<NX>(y2, g, nl, x, v[e]);
      norm_add(b, s[0]);
      norm_add(v[e], s[2]);
    });
  }
  __syncthreads();  // the tile is free
  block_sums(s, reinterpret_cast<double*>(smem_raw), [&](int k, double t) { a.part[(long long)k * a.stride + blockIdx.x] = t; });
}

template <typename Real> cudaError_t launch_gs_fwd(int nx, const GsFwd& a, const void* twn, cudaStream_t st);
template <typename Real> cudaError_t launch_gs_inv(int nx, const GsInv& a, const void* twn, cudaStream_t st);

#ifdef FSE_GSX_INSTANTIATE
template <typename Real, int NX, int LN>
static cudaError_t gs_fwd_launch(const GsFwd& a, const void* twn, cudaStream_t st) {
  typedef XCfg<Real, NX, LN> K;
  typedef const typename TwOf<Real>::T* W;
  static std::atomic<unsigned long long> done0{0}, done1{0};
  cudaError_t e = a.dy ? allow_smem(k_gs_fwd<Real, NX, LN, true>, K::smem(), done1)
                       : allow_smem(k_gs_fwd<Real, NX, LN, false>, K::smem(), done0);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (a.nlines + LN - 1) / LN;
  return a.dy ? launch_pass(k_gs_fwd<Real, NX, LN, true>, blocks, K::NT, K::smem(), st, a, reinterpret_cast<W>(twn))
              : launch_pass(k_gs_fwd<Real, NX, LN, false>, blocks, K::NT, K::smem(), st, a, reinterpret_cast<W>(twn));
}
template <typename Real, int NX, int LN>
static cudaError_t gs_inv_launch(const GsInv& a, const void* twn, cudaStream_t st) {
  typedef XCfg<Real, NX, LN> K;
  const size_t smem = K::smem() > 32 * (size_t)K::NT ? K::smem() : 32 * (size_t)K::NT;  // the tile, or four sums per thread
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_gs_inv<Real, NX, LN>, smem, done);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (a.nlines + LN - 1) / LN;
  return launch_pass(k_gs_inv<Real, NX, LN>, blocks, K::NT, smem, st, a,
                     reinterpret_cast<const typename TwOf<Real>::T*>(twn));
}
template <typename Real> cudaError_t launch_gs_fwd(int nx, const GsFwd& a, const void* twn, cudaStream_t st) {
  switch (nx) {
#define FSE_CASE(n)                                                                \
  case n:                                                                          \
    return xpass_pick<Real, n>(a.nlines, 1) == XWidths<Real, n>::wide()            \
               ? gs_fwd_launch<Real, n, XWidths<Real, n>::wide()>(a, twn, st)      \
               : gs_fwd_launch<Real, n, XWidths<Real, n>::narrow()>(a, twn, st);
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}
template <typename Real> cudaError_t launch_gs_inv(int nx, const GsInv& a, const void* twn, cudaStream_t st) {
  switch (nx) {
#define FSE_CASE(n)                                                                \
  case n:                                                                          \
    return xpass_pick<Real, n>(a.nlines, 1) == XWidths<Real, n>::wide()            \
               ? gs_inv_launch<Real, n, XWidths<Real, n>::wide()>(a, twn, st)      \
               : gs_inv_launch<Real, n, XWidths<Real, n>::narrow()>(a, twn, st);
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}
#endif

}  // namespace fse
