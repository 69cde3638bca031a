// fse_col.cuh -- column passes: transforms along a strided axis (y or z), tiles of adjacent columns.
//
// Variants (VAR), n the axis's length:
//   COL_FWD / COL_INV  one transform of the wave function (exact twiddles)
//   COL_KIN            fwd . kinetic phase . inv of the wave function
//   COL_PADF           forward transform of n rows zero-padded to 2n (density)
//   COL_CROPI          inverse transform of 2n rows keeping rows [0, n) (density)
//   COL_KHAT           n rows zero-padded to 2n, fwd . kernel transform . inv, rows [0, n) kept
//   COL_KIN2 / COL_KHAT2  the same on the y axis of a 2D grid
//   COL_RMUL           fwd . real spectral factor . inv (ground state)
//   COL_DY             fwd . i k . inv, out of place (derivative along the axis)
//   COL_LZ             the same derivative d of psi, not stored: partials of sum x Im(conj(psi) d)
// The padded variants transform length 2n: their first pass leaves out the
// zero half of its inputs, their last one computes only the rows that are kept.
#pragma once

#include "fse_vec.cuh"

namespace fse {

enum { MUL_KIN = 1, MUL_COULOMB = 2, MUL_DDI = 3 };
enum { COL_FWD = 0, COL_INV = 1, COL_PADF = 2, COL_CROPI = 3, COL_KIN = 4, COL_KHAT = 5, COL_KIN2 = 6, COL_KHAT2 = 7, COL_RMUL = 8, COL_DY = 9, COL_LZ = 10 };

struct ColArgs {
  void* data;
  long long plane_stride;  // elements between planes
  long long line_stride;   // elements between consecutive points of a line
  int nplanes, ncols;      // planes; columns (lines) per plane, contiguous
  // set by the launch: tiles_per_plane full tiles of every plane; tail > 0:
  // they cover the first tiles_per_plane * NC columns, and further tiles each
  // take NC consecutive (plane, column) pairs of the `tail` remaining columns
  int tiles_per_plane, tail;
  void* out;  // COL_DY: the result's buffer
  double* part;     // COL_LZ: one partial per block
  double lo, h;     // COL_LZ: coordinate of column i, lo + h i
  int* blocks_out;  // host: receives the number of blocks (null: not wanted)
};

struct MulArgs {
  int mode;
  int lx;            // signed-wrap length of the column (x) index; 0 = R2C bin (non-negative)
  int lp;            // signed-wrap length of the plane index (0 = no plane axis)
  double dkr;        // COL_DY, COL_LZ: spacing of the axis over its length
  double scale;      // 1/N of the transform
  double a0;         // Coulomb: dt*scale; DDI: -dt*scale
  double q[6];       // DDI: 3*scale*(Mxx, Mpp, Mrr, 2 Mxp, 2 Mxr, 2 Mpr) times the two axes' spacings
  const void* chat;
  long long chat_sp, chat_sr;
  int chat_cx;       // padded length of a C^ row (x bins 0..lx/2, then zeros), a multiple of 4
  const void* kin;   // COL_RMUL: octant table of real factors; kinetic: octant table of exp(-i f theta_k) on |p_j| = 0..n_j/2
  long long kin_sp, kin_sr;  // kinetic: octant strides of the plane and row axes
  int conj;          // kinetic: multiply by the conjugate of the table (adjoint)
  // float copies of the scalars above, written by fill_f32 before a launch: a
  // float kernel reads them as they are instead of converting the double
  // fields in every thread (double-to-float conversions issue on the narrow
  // FP64 pipe)
  struct {
    float dkr, scale, a0, q[6], qt[6];  // qt: what rounding q to float leaves
  } f;
};

__host__ __device__ inline void fill_f32(MulArgs& m) {
  m.f.dkr = (float)m.dkr;
  m.f.scale = (float)m.scale;
  m.f.a0 = (float)m.a0;
  for (int i = 0; i < 6; ++i) {
    m.f.q[i] = (float)m.q[i];
    m.f.qt[i] = (float)(m.q[i] - (double)m.f.q[i]);
  }
}

// A scalar parameter in the kernel's precision: the double field, or its float copy.
template <typename Real>
__device__ __forceinline__ Real prm(double d, float f);
template <> __device__ __forceinline__ float prm<float>(double, float f) { return f; }
template <> __device__ __forceinline__ double prm<double>(double d, float) { return d; }

__device__ __forceinline__ int wrap_index(int i, int L) { return i < (L >> 1) ? i : i - L; }

// First statement of every step pass. The passes of a step are launched with
// programmatic dependent launch: a block waits here until the previous pass has
// completed and its writes are visible (immediate for a launch without that
// dependency). No pass lets the next one be launched before its own blocks end
// (griddepcontrol.launch_dependents): blocks that are launched among those of a
// running pass are dealt to the SMs by the room they find there, and an SM that
// gets a few too many sets the time (192 float64 tiles of 64 points 20 us
// instead of 3.6, 256 float32 ones of 96 points 14 instead of 6.6). The launch's
// latency is hidden all the same. Two steps of 128^3 float32 239 -> 215 us, of
// 256^2 float64 139 -> 127; 500 calls of all kinds and sizes 6 % less on average,
// the shortest ground states and shifts (32^3) 4 to 12 % more.
__device__ __forceinline__ void pass_prologue() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

constexpr int kSMs = 152;  // GB300

// Shape of a column pass along an axis of N points; THIN: of its narrower tiles.
template <typename Real, int N, int VAR, bool THIN = false>
struct ColShape {
  typedef typename LaneOf<Real>::T L;
  static constexpr int CW = sizeof(L) / sizeof(Real);  // columns per 16-byte element
  static constexpr bool KIN = VAR == COL_KIN || VAR == COL_KIN2, KHAT = VAR == COL_KHAT || VAR == COL_KHAT2;
  static constexpr bool TWO = VAR == COL_PADF || VAR == COL_CROPI || KHAT;  // length 2N
  static constexpr int M = TWO ? 2 * N : N;
  static constexpr bool EXACT = !TWO;
  // Float plans. 3D passes have planes enough to fill the SMs with any tile
  // and are bound by issue: the large radices (256^3: pass C 82 us against 92
  // with 8 x 8 x 4; pass G with two items of eight elements per thread 233 us
  // against 252 with one). A 2D grid is one plane: a single run's time is the
  // latency of a thread's chain, which eight elements per thread halve (one
  // 256^2 run: kinetic pass 7.8 -> 7.1 us, kernel pass 5.7 -> 4.2 us; batched
  // 256^2 runs: 40.4 -> 37.4 and 40.7 -> 37.9 us per 50 runs). Length 96 takes
  // the eight-element plan everywhere (12 x 8 leaves a third of the threads
  // idle while the tile is loaded), and so do the shortest axes.
  // Narrow tiles are a chain of latencies too: theirs is the plan of at most
  // eight elements, with a thread for every item of radix 4 or more (2D passes
  // keep their radices, so that a run's bits do not depend on how many advance
  // together). Two steps: 16 x 16 x 128 39 -> 32 us, 12 x 64 x 24 58 -> 50, 256^2
  // without interaction 38 -> 32, 192 x 96 55 -> 46.
  static constexpr bool D2 = VAR == COL_KIN2 || VAR == COL_KHAT2;
  static constexpr bool SLIM2 = VAR == COL_KIN2 || (VAR == COL_KHAT2 && M <= 256);
  static constexpr bool SLIM = SLIM2 || (!TWO && M == 96) || N <= 32 || (THIN && !D2);
  __host__ __device__ static constexpr int threads() {
    if (sizeof(Real) == 8) return 0;
    if (!THIN) return M == 512 && VAR == COL_KHAT ? 32 : 0;
    if (D2 && !SLIM2) return 0;
    const FftPlan p = fft_plan_slim(M);
    int r = p.r[0];
    for (int i = 1; i < p.np; ++i) r = p.r[i] < r ? p.r[i] : r;
    const int t = M / (r < 4 ? 4 : r);
    return t < p.T || t > 128 ? p.T : t;
  }
  typedef FftCfg<Real, M, threads(), SLIM> F;
  static constexpr int T = F::T;
  // Tile widths in elements: wide tiles move rows of 128 (64) bytes; the
  // narrow one is as few columns as still fill a warp, for grids whose wide
  // tiles would leave SMs idle.
  __host__ __device__ static constexpr int wide() {
    if (T * 8 < 32) return 32 / T;
    if (T >= 128) return 512 / T;
    if (sizeof(Real) == 8) return T >= 48 ? 4 : 8;
    return T >= 64 && (M != 512 || KHAT) ? 4 : 8;
  }
  __host__ __device__ static constexpr int narrow() {
    int w = 1;
    while (w * ColShape<Real, N, VAR, true>::T < 32) w *= 2;
    return w < wide() ? w : wide();
  }
  // between the two where they lie far apart
  __host__ __device__ static constexpr int mid() { return wide() >= 4 * narrow() ? wide() / 2 : wide(); }
};

template <typename Real, int N, int VAR, int NP>
struct ColCfg {
  static constexpr int WIDE = ColShape<Real, N, VAR>::wide();
  typedef ColShape<Real, N, VAR, (NP < WIDE)> S;
  typedef typename S::F F;
  static constexpr int M = S::M, T = S::T, NT = NP * T, E = F::E;
  static constexpr int NC = S::CW * NP;  // columns per tile
  // rows of 8 or more slots need no padding (a quarter warp touches one row);
  // narrower ones skip a row after every FR rows, FR the first radix
  static constexpr bool PAD = NP < 8;
  static constexpr int MINR = F::RF < F::RL ? F::RF : F::RL;
  static constexpr size_t EXCH = F::P.np > 1 ? 16 * (size_t)NP * (M + (PAD ? M / MINR : 0)) : 0;
  static constexpr size_t CHAT = S::KHAT ? sizeof(Real) * (size_t)(N + 1) * NC : 0;
  __host__ __device__ static constexpr size_t smem() { return EXCH + CHAT; }
  // registers: 128 per thread for 16 float pairs (64 data registers) and the
  // float64 passes with eight elements, 96 up to 12 elements, 80 or 64 below.
  __host__ __device__ static constexpr int minb() {
    const int thr = E > 12 || (sizeof(Real) == 8 && E > 6) ? 512
                                                           : (E > 8 || sizeof(Real) == 8 || VAR == COL_LZ ? 640 : (S::KHAT ? 768 : 1024));
    const int b = thr / ((NT + 31) / 32 * 32);
    return b < 1 ? 1 : (b > 32 ? 32 : b);
  }
};

// Address map of a column tile and its barrier.
template <int NP, bool PAD> struct ColAddr {
  int g;
  template <int FR> __device__ __forceinline__ int slot(int row) const {
    if constexpr (PAD) return (row + row / FR) * NP + g;
    else return row * NP + g;
  }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};

// This thread's columns (CW of them): plane, x index, validity, base pointer.
template <typename Real, int CW> struct ColGeo {
  typedef typename Cplx<Real>::T C;
  int plane[CW], px[CW];
  bool ok[CW];
  C* p[CW];
  bool vec;  // float: both columns valid, adjacent and 16-byte aligned, one access per row
};

template <int CW>
__device__ __forceinline__ Vec<float2> col_ld(const ColGeo<float, CW>& g, unsigned o) {
  if (g.vec) {
    const float4 t = *reinterpret_cast<const float4*>(g.p[0] + o);
    return {make_float2(t.x, t.z), make_float2(t.y, t.w)};
  }
  const float2 z = make_float2(0.f, 0.f);
  const float2 a = g.ok[0] ? g.p[0][o] : z, b = g.ok[1] ? g.p[1][o] : z;
  return {make_float2(a.x, b.x), make_float2(a.y, b.y)};
}
template <int CW>
__device__ __forceinline__ void col_st(const ColGeo<float, CW>& g, unsigned o, const Vec<float2>& v) {
  if (g.vec) {
    *reinterpret_cast<float4*>(g.p[0] + o) = make_float4(v.re.x, v.im.x, v.re.y, v.im.y);
  } else {
    if (g.ok[0]) g.p[0][o] = make_float2(v.re.x, v.im.x);
    if (g.ok[1]) g.p[1][o] = make_float2(v.re.y, v.im.y);
  }
}
template <int CW>
__device__ __forceinline__ Vec<double> col_ld(const ColGeo<double, CW>& g, unsigned o) {
  if (!g.ok[0]) return {0.0, 0.0};
  const double2 t = g.p[0][o];
  return {t.x, t.y};
}
template <int CW>
__device__ __forceinline__ void col_st(const ColGeo<double, CW>& g, unsigned o, const Vec<double>& v) {
  if (g.ok[0]) g.p[0][o] = make_double2(v.re, v.im);
}

// Product with a kinetic factor (c + i s per column, conjugated for the
// adjoint) and the transform's 1/N; float: the pair's modulus error is folded
// into the products before their final rounding (unit_mul).
__device__ __forceinline__ Vec<float2> kin_mul(const Vec<float2>& x, const float2 (&t)[2], bool conj, float scale) {
  const float2 c = make_float2(t[0].x, t[1].x);
  const float2 s = conj ? make_float2(-t[0].y, -t[1].y) : make_float2(t[0].y, t[1].y);
  const float2 h = make_float2(-0.5f * norm_err(t[0].x, t[0].y), -0.5f * norm_err(t[1].x, t[1].y));
  const float2 lc = lmul(h, c), ls = lmul(h, s), sc = make_float2(scale, scale);
  const float2 lr = lfma(x.re, lc, lmul(x.im, lneg(ls)));
  const float2 li = lfma(x.re, ls, lmul(x.im, lc));
  return {lmul(sc, lfma(x.re, c, lfma(x.im, lneg(s), lr))), lmul(sc, lfma(x.re, s, lfma(x.im, c, li)))};
}
__device__ __forceinline__ Vec<double> kin_mul(const Vec<double>& x, const double2 (&t)[1], bool conj, double scale) {
  const double c = scale * t[0].x, s = conj ? -scale * t[0].y : scale * t[0].y;
  return {lfma(x.re, c, lmul(x.im, -s)), lfma(x.re, s, lmul(x.im, c))};
}

__device__ __forceinline__ float2 lane_of(const float (&v)[2]) { return make_float2(v[0], v[1]); }
__device__ __forceinline__ double lane_of(const double (&v)[1]) { return v[0]; }
__device__ __forceinline__ float2 lane_ld(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ double lane_ld(const double* p) { return *p; }

// Head and tail: the exact product of two lanes, and sums good to the square of
// the rounding unit.
template <typename L> struct Two {
  L h, l;
};
template <typename L> __device__ __forceinline__ Two<L> two_prod(L a, L b) {
  const L p = lmul(a, b);
  return {p, lfma(a, b, lneg(p))};
}
template <typename L> __device__ __forceinline__ Two<L> two_sum(const Two<L>& a, const Two<L>& b) {
  const L s = ladd(a.h, b.h), v = lsub(s, a.h);
  const L e = ladd(lsub(a.h, lsub(s, v)), lsub(b.h, v));
  return {s, ladd(e, ladd(a.l, b.l))};
}

// s += Im(conj(u) d), u scaled by su and d by sd
template <typename L>
__device__ __forceinline__ void lz_add(const Vec<L>& u, const Vec<L>& d, const L& su, const L& sd, ExactSum<L>& s) {
  const L re = lmul(su, u.re), im = lneg(lmul(su, u.im));
  s.prod(re, lmul(sd, d.im));
  s.prod(im, lmul(sd, d.re));
}
// max modulus of the components of the elements a thread holds before (after)
// the transforms; a length that leaves threads short of items leaves elements unset
template <typename F, typename L, int E> __device__ __forceinline__ float vmax_abs(int it, const Vec<L> (&v)[E]) {
  float m = 0.f;
  F::template each<F::RF>(it, [&](int e, int, int) { m = lmax_abs(lmax_abs(m, v[e].re), v[e].im); });
  return m;
}

template <typename Real, int N, int VAR, int NP, bool GATHER, bool PDL>
__device__ __forceinline__ void col_tile(const ColArgs& a, const MulArgs& m, const typename TwOf<Real>::T* __restrict__ tw,
                                         int bid, int ngat) {
  typedef ColCfg<Real, N, VAR, NP> K;
  typedef typename K::F F;
  typedef typename LaneOf<Real>::T L;
  typedef typename Cplx<Real>::T C;
  constexpr int CW = K::S::CW, NC = K::NC, NT = K::NT, M = K::M, RF = F::RF, RL = F::RL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* buf = reinterpret_cast<float4*>(smem_raw);
  Real* sC = reinterpret_cast<Real*>(smem_raw + K::EXCH);
  const int tid = threadIdx.x;
  int it = tid / NP;
  const ColAddr<NP, K::PAD> addr{tid % NP};
  const unsigned ls = (unsigned)a.line_stride;  // a plane's elements fit 32 bits
  // hides that `it` is unchanged, so that addresses are computed again rather
  // than held in registers across a whole transform
  auto fresh = [&]() { asm volatile("" : "+r"(it)); };

  // columns of this thread
  const int breg = bid - ngat;
  const int tp = GATHER ? 0 : breg / a.tiles_per_plane;
  const int c0 = GATHER ? 0 : (breg - tp * a.tiles_per_plane) * NC;
  // kernel-transform pass over a full even set of planes: planes p and lp - p
  // (same |p|, same C^ values) run next to each other, so the octant is read
  // from HBM about once
  const int plane = (K::S::KHAT && m.lp == a.nplanes && (m.lp & 1) == 0 && tp > 0)
                        ? ((tp & 1) ? (tp + 1) >> 1 : m.lp - (tp >> 1))
                        : tp;
  ColGeo<Real, CW> geo;
#pragma unroll
  for (int q = 0; q < CW; ++q) {
    const int cc = addr.g * CW + q;
    if constexpr (!GATHER) {
      geo.plane[q] = plane;
      geo.px[q] = c0 + cc;
      geo.ok[q] = geo.px[q] < a.ncols;
    } else {
      const int qq = bid * NC + cc;
      geo.plane[q] = qq / a.tail;
      geo.px[q] = a.tiles_per_plane * NC + qq % a.tail;
      geo.ok[q] = geo.plane[q] < a.nplanes;
      if (!geo.ok[q]) geo.plane[q] = geo.px[q] = 0;
    }
    geo.p[q] = (!GATHER && q > 0) ? geo.p[0] + q
                                  : reinterpret_cast<C*>(a.data) + (long long)geo.plane[q] * a.plane_stride + geo.px[q];
  }
  // Tiles narrower than the widest are the only ones on their SM, and a pass is
  // then a chain of memory latencies. The constant tables it will read (twiddles,
  // kinetic factors, C^) come into L1 or shared memory before the wait for the
  // previous pass, which they do not depend on.
  constexpr bool EARLY = PDL && NP < K::WIDE;
  if constexpr (EARLY && F::P.np > 1) {
    unsigned x = F::template warm_table<VAR == COL_CROPI, K::S::EXACT, NT>(tw, tid);
    if constexpr (K::S::KIN || K::S::KHAT) x ^= F::template warm_table<true, K::S::EXACT, NT>(tw, tid);
    if constexpr (K::S::KIN) {
      const C* t = reinterpret_cast<const C*>(m.kin) + (m.lp ? (long long)abs(wrap_index(geo.plane[0], m.lp)) * m.kin_sp : 0) +
                   abs(wrap_index(min(geo.px[0], m.lx - 1), m.lx));
      unsigned w[N / 2 / F::T + 1];
#pragma unroll
      for (int i = 0; i <= N / 2 / F::T; ++i) w[i] = warm_line(t + min(it + i * F::T, N / 2) * m.kin_sr);
#pragma unroll
      for (int i = 0; i <= N / 2 / F::T; ++i) x ^= w[i];
    }
    reinterpret_cast<unsigned*>(smem_raw)[tid] = x;
  }
  if constexpr (PDL && !(EARLY && K::S::KHAT)) pass_prologue();
  geo.vec = !GATHER && CW == 2 && geo.ok[CW - 1] && (reinterpret_cast<uintptr_t>(geo.p[0]) % 16 == 0) &&
            (a.line_stride % 2 == 0);

  if constexpr (K::S::KHAT) {
    // the tile's C^ values (|p_row| = 0..N) into shared memory while the first transform runs
    const Real* ch = reinterpret_cast<const Real*>(m.chat);
    if constexpr (!GATHER) {
      // the tile's columns of a C^ row are contiguous and aligned (rows padded
      // to a multiple of 4 values, c0 a multiple of NC); copies past the
      // padded row are zero-filled
      constexpr int EPC = (NC * (int)sizeof(Real) >= 16 ? 16 : NC * (int)sizeof(Real)) / (int)sizeof(Real), CPR = NC / EPC;
      static_assert(NC % EPC == 0, "C^ copies");
      const Real* chp = ch + (m.lp ? (long long)abs(wrap_index(plane, m.lp)) * m.chat_sp : 0) + c0;
      const int left = m.chat_cx - c0;
      for (int idx = tid; idx < (N + 1) * CPR; idx += NT) {
        const int ar = idx / CPR, qd = idx - ar * CPR;
        Real* dst = &sC[ar * NC + qd * EPC];
        if (qd * EPC < left) {
          cp_async<EPC * (int)sizeof(Real)>(dst, &chp[(long long)ar * m.chat_sr + qd * EPC]);
        } else {
#pragma unroll
          for (int e = 0; e < EPC; ++e) dst[e] = Real(0);
        }
      }
    } else {
      for (int idx = tid; idx < (N + 1) * NC; idx += NT) {
        const int ar = idx / NC, qq = bid * NC + idx % NC;
        const int pl = qq / a.tail, px = a.tiles_per_plane * NC + qq % a.tail;
        if (pl < a.nplanes && px <= (m.lx >> 1))
          cp_async<sizeof(Real)>(&sC[idx], &ch[(long long)ar * m.chat_sr +
                                               (m.lp ? (long long)abs(wrap_index(pl, m.lp)) * m.chat_sp : 0) + px]);
        else
          sC[idx] = Real(0);
      }
    }
    cp_async_commit();
  }
  if constexpr (EARLY && K::S::KHAT) pass_prologue();
  if constexpr (EARLY) __syncthreads();  // the warm-up's words are written before the tile is

  Vec<L> v[F::E];
  if constexpr (VAR == COL_FWD || VAR == COL_INV) {
    F::template each<RF>(it, [&](int e, int row, int) { v[e] = col_ld(geo, row * ls); });
    F::template run<VAR == COL_INV ? +1 : -1, true, false, false>(v, buf, addr, tw, it);
    fresh();
    F::template each<RL>(it, [&](int e, int row, int) { col_st(geo, row * ls, v[e]); });
  } else if constexpr (VAR == COL_PADF) {
    F::template each<RF>(it, [&](int e, int row, int r) {
      if (2 * r < RF) v[e] = col_ld(geo, row * ls);
    });
    F::template run<-1, false, false, false, true>(v, buf, addr, tw, it);
    fresh();
    F::template each<RL>(it, [&](int e, int row, int) { col_st(geo, row * ls, v[e]); });
  } else if constexpr (VAR == COL_CROPI) {
    // the radices in reverse, so that the rows kept are outputs r < RF/2 of every item
    F::template each<RL>(it, [&](int e, int row, int) { v[e] = col_ld(geo, row * ls); });
    F::template run<+1, false, true, false>(v, buf, addr, tw, it);
    fresh();
    F::template each<RF>(it, [&](int e, int row, int r) {
      if (2 * r < RF) col_st(geo, row * ls, v[e]);
    });
  } else if constexpr (VAR == COL_RMUL) {
    F::template each<RF>(it, [&](int e, int row, int) { v[e] = col_ld(geo, row * ls); });
    F::template run<-1, true, false, false>(v, buf, addr, tw, it);
    const Real* tab[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q)
      tab[q] = reinterpret_cast<const Real*>(m.kin) +
               (m.lp ? (long long)abs(wrap_index(geo.plane[q], m.lp)) * m.kin_sp : 0) +
               abs(wrap_index(min(geo.px[q], m.lx - 1), m.lx));
    fresh();
    F::template each<RL>(it, [&](int e, int row, int) {
      const long long ro = (long long)abs(wrap_index(row, N)) * m.kin_sr;
      Real t[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) t[q] = __ldg(&tab[q][ro]);
      const L f = lane_of(t);
      v[e] = {lmul(f, v[e].re), lmul(f, v[e].im)};
    });
    fresh();
    F::template run<+1, true, true, true>(v, buf, addr, tw, it);
    fresh();
    F::template each<RF>(it, [&](int e, int row, int) { col_st(geo, row * ls, v[e]); });
  } else if constexpr (VAR == COL_DY || VAR == COL_LZ) {
    F::template each<RF>(it, [&](int e, int row, int) { v[e] = col_ld(geo, row * ls); });
    float um = 0.f;
    if constexpr (VAR == COL_LZ) um = vmax_abs<F>(it, v);
    F::template run<-1, true, false, false>(v, buf, addr, tw, it);
    const Real dk = prm<Real>(m.dkr, m.f.dkr);  // includes 1/N
    F::template each<RL>(it, [&](int e, int row, int) {
      // the odd factor is zero at the Nyquist index
      const L k = lbc<L>(2 * row == N ? Real(0) : dk * Real(wrap_index(row, N)));
      v[e] = {lneg(lmul(k, v[e].im)), lmul(k, v[e].re)};
    });
    F::template run<+1, true, true, true>(v, buf, addr, tw, it);
    fresh();
    if constexpr (VAR == COL_LZ) {
      __shared__ double red[32];
      // (the thread's rows here are the ones it loaded at first)
      const Pow2<L> su = pow2_scale<L>(um), sd = pow2_scale<L>(vmax_abs<F>(it, v));
      ExactSum<L> s;
      F::template each<RF>(it, [&](int e, int row, int) { lz_add(col_ld(geo, row * ls), v[e], su.scale, sd.scale, s); });
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < CW; ++q)
        if (geo.ok[q]) t += (a.lo + a.h * geo.px[q]) * s.get(q);
      t *= su.inv * sd.inv;
      t = block_sum(t, red);
      if (tid == 0) a.part[bid] = t;
    } else {
#pragma unroll
      for (int q = 0; q < CW; ++q) geo.p[q] = reinterpret_cast<C*>(a.out) + (geo.p[q] - reinterpret_cast<C*>(a.data));
      geo.vec = geo.vec && (reinterpret_cast<uintptr_t>(geo.p[0]) % 16 == 0);
      F::template each<RF>(it, [&](int e, int row, int) { col_st(geo, row * ls, v[e]); });
    }
  } else if constexpr (K::S::KIN) {
    F::template each<RF>(it, [&](int e, int row, int) { v[e] = col_ld(geo, row * ls); });
    F::template run<-1, true, false, false>(v, buf, addr, tw, it);
    // kinetic phase exp(-i f theta_k) from the plan's octant table, indexed by
    // |p_x| (column), |p_plane| and |p_row| (row = frequency index along the
    // axis), on the outputs as they sit in registers; the inverse takes the
    // radices in reverse order and starts on them
    const C* tab[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q)
      tab[q] = reinterpret_cast<const C*>(m.kin) + (m.lp ? (long long)abs(wrap_index(geo.plane[q], m.lp)) * m.kin_sp : 0) +
               abs(wrap_index(min(geo.px[q], m.lx - 1), m.lx));
    fresh();
    const Real sc = prm<Real>(m.scale, m.f.scale);
    const bool conj = m.conj != 0;
    F::template each<RL>(it, [&](int e, int row, int) {
      const long long ro = (long long)abs(wrap_index(row, N)) * m.kin_sr;
      C t[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) t[q] = __ldg(&tab[q][ro]);
      v[e] = kin_mul(v[e], t, conj, sc);
    });
    fresh();
    F::template run<+1, true, true, true>(v, buf, addr, tw, it);
    fresh();
    F::template each<RF>(it, [&](int e, int row, int) { col_st(geo, row * ls, v[e]); });
  } else {
    F::template each<RF>(it, [&](int e, int row, int r) {
      if (2 * r < RF) v[e] = col_ld(geo, row * ls);
    });
    F::template run<-1, false, false, false, true>(v, buf, addr, tw, it);
    // kernel transform on the padded grid: f = a0 C^ (Coulomb) or a0 + (k^T Q k) C^
    // (DDI); the column (x, an R2C bin 0..nx) and plane factors are fixed per thread
    cp_async_wait_all();
    addr.sync();
    fresh();
    const bool ddi = m.mode == MUL_DDI;
    // integer frequencies: the spacings are in the factors q. A and B are one
    // value for a column, and the dipolar energy is a small difference of sums over
    // all modes: float plans form both as sums of two floats, with what rounding the
    // factors left, and A's tail goes on to the elements (rounded in every product
    // the columns alone left 1e-8 to 2e-8 of the two sums in the energy; now 4e-9.
    // 256^3 3299 us for four steps without the tails of A, 3310 with them)
    L A = lbc<L>(0.0), B = A, Al = A;
    if (ddi) {
      Real kp_[CW], kx_[CW], kpo_[CW], kxo_[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) {
        kp_[q] = m.lp ? Real(wrap_index(geo.plane[q], m.lp)) : Real(0);
        kpo_[q] = (m.lp && 2 * geo.plane[q] == m.lp) ? Real(0) : kp_[q];
        kx_[q] = Real(geo.px[q]);
        kxo_[q] = (2 * geo.px[q] == m.lx) ? Real(0) : kx_[q];
      }
      const L kp = lane_of(kp_), kx = lane_of(kx_), kpo = lane_of(kpo_), kxo = lane_of(kxo_);
      const L xx = lmul(kx, kx), pp = lmul(kp, kp), xp = lmul(kxo, kpo);  // (exact)
      auto q = [&](int i) { return lbc<L>(prm<Real>(m.q[i], m.f.q[i])); };
      if constexpr (sizeof(Real) == 4) {
        auto t = [&](int i) { return lbc<L>(m.f.qt[i]); };
        const Two<L> a = two_sum(two_sum(two_prod(q(0), xx), two_prod(q(1), pp)), two_prod(q(3), xp));
        const L al = lfma(t(0), xx, lfma(t(1), pp, lfma(t(3), xp, a.l)));
        A = ladd(a.h, al);
        Al = lsub(al, lsub(A, a.h));
        const Two<L> b = two_sum(two_prod(q(4), kxo), two_prod(q(5), kpo));
        B = ladd(b.h, lfma(t(4), kxo, lfma(t(5), kpo, b.l)));
      } else {
        A = lfma(q(0), xx, lfma(q(1), pp, lmul(q(3), xp)));
        B = lfma(q(4), kxo, lmul(q(5), kpo));
      }
    }
    const L a0 = lbc<L>(prm<Real>(m.a0, m.f.a0));
    const L q2 = lbc<L>(prm<Real>(m.q[2], m.f.q[2]));
    F::template each<RL>(it, [&](int e, int row, int r) {
      // signed frequency of the row: row - M from M/2 on
      const bool up = RL % 2 == 0 ? 2 * r >= RL : 2 * row >= M;
      const L cv = lane_ld(&sC[(up ? M - row : row) * NC + addr.g * CW]);
      if (ddi) {
        // an exact sum of small integers; the first is the same for every r of an item
        const L kr = lbc<L>(Real(row - r * (M / RL)) + Real(r * (M / RL) - (up ? M : 0)));
        L b = 2 * row == M ? lbc<L>(0.0) : B;
        if constexpr (sizeof(Real) == 4) b = lfma(lbc<L>(m.f.qt[2]), kr, b);
        L f0 = a0;
        if constexpr (sizeof(Real) == 4) f0 = lfma(Al, cv, a0);
        const L f = lfma(lfma(kr, lfma(q2, kr, b), A), cv, f0);
        v[e] = {lmul(f, v[e].re), lmul(f, v[e].im)};
      } else {
        const L f = lmul(a0, cv);
        v[e] = {lmul(f, v[e].re), lmul(f, v[e].im)};
      }
    });
    fresh();
    F::template run<+1, false, true, true>(v, buf, addr, tw, it);
    fresh();
    F::template each<RF>(it, [&](int e, int row, int r) {
      if (2 * r < RF) col_st(geo, row * ls, v[e]);
    });
  }
}

// One tile of a column pass (block bid). Passes over R2C bins gather the bin
// n_x of all planes into the first tiles of the grid, so that they overlap the
// full tiles; the two kinds are separate instantiations, so that the per-column
// state of the gathered tiles does not take registers from the full ones.
// PDL: the launch is a dependent one (the prologue's wait is here).
template <typename Real, int N, int VAR, int NP, bool PDL>
__device__ __forceinline__ void col_body(const ColArgs& a, const MulArgs& m, const typename TwOf<Real>::T* __restrict__ tw,
                                         int bid) {
  typedef ColCfg<Real, N, VAR, NP> K;
  if constexpr (K::S::TWO && VAR != COL_KHAT2) {  // (a 2D pass is one plane: nothing to gather)
    const int ngat = a.tail > 0 ? (a.nplanes * a.tail + K::NC - 1) / K::NC : 0;
    if (bid < ngat) col_tile<Real, N, VAR, NP, true, PDL>(a, m, tw, bid, ngat);
    else col_tile<Real, N, VAR, NP, false, PDL>(a, m, tw, bid, ngat);
  } else {
    col_tile<Real, N, VAR, NP, false, PDL>(a, m, tw, bid, 0);
  }
}

template <typename Real, int N, int VAR, int NP>
__global__ void __launch_bounds__(ColCfg<Real, N, VAR, NP>::NT, ColCfg<Real, N, VAR, NP>::minb())
k_col(ColArgs a, MulArgs m, const typename TwOf<Real>::T* __restrict__ tw) {
  col_body<Real, N, VAR, NP, true>(a, m, tw, blockIdx.x);
}

// Tiles of NC columns over the passes' planes; returns the blocks. Passes over
// the R2C bins 0..nx of many planes: the last, nearly empty tile of every
// plane (nx + 1 = k NC + 1 bins for the usual sizes) is replaced by tail tiles
// holding that column of NC planes each.
inline long long col_tiles(ColArgs& a, int nc, bool tails) {
  const int rem = a.ncols % nc;
  a.tail = 0;
  a.tiles_per_plane = (a.ncols + nc - 1) / nc;
  if (tails && a.nplanes > 1 && rem > 0 && 2 * rem <= nc && a.ncols >= nc) {
    a.tiles_per_plane = a.ncols / nc;
    a.tail = rem;
  }
  return (long long)a.nplanes * a.tiles_per_plane + (a.tail > 0 ? ((long long)a.nplanes * a.tail + nc - 1) / nc : 0);
}

// Launch of one variant of the pass along an axis of n points: tw the twiddle
// table of the pass's length, 2n for the padded variants.
template <typename Real, int VAR>
cudaError_t launch_col_var(int n, const ColArgs& a, const MulArgs& m, const void* tw, cudaStream_t st);

}  // namespace fse
