// fse_launch.cuh -- size dispatch of the pass kernels (included by one .cu per precision and kind).
#pragma once

#include <atomic>
#include <type_traits>

#include "fse_passes.cuh"

namespace fse {

// Grid lengths.
#define FSE_SIZES(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512)

// Launch of a step pass with programmatic dependent launch on the previous
// kernel in the stream (see pass_prologue).
template <typename... Params, typename... Args>
static cudaError_t launch_pass(void (*kernel)(Params...), unsigned blocks, unsigned threads, size_t smem,
                               cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// cudaFuncSetAttribute once per kernel and device when the dynamic tile comes
// near the 48 KB default (the kernels also hold up to 1 KB of static shared memory).
template <typename F>
static cudaError_t allow_smem(F* fn, size_t bytes, std::atomic<unsigned long long>& done) {
  if (bytes + 1024 <= 48 * 1024) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load() & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) done.fetch_or(bit);
  return e;
}

template <typename Real, int N, int VAR, int NP>
static cudaError_t col_launch(const ColArgs& a, const MulArgs& m, long long blocks, const void* tw,
                              cudaStream_t st) {
  typedef ColCfg<Real, N, VAR, NP> K;
  typedef typename TwOf<Real>::T C;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_col<Real, N, VAR, NP>, K::smem(), done);
  if (e != cudaSuccess) return e;
  if (blocks <= 0) return cudaSuccess;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (a.blocks_out) *a.blocks_out = (int)blocks;
  MulArgs mf = m;
  fill_f32(mf);
  return launch_pass(k_col<Real, N, VAR, NP>, (unsigned)blocks, K::NT, K::smem(), st, a, mf,
                     reinterpret_cast<const C*>(tw));
}

// The width of a column pass's tiles: the widest whose tiles give every SM
// one, else the narrowest: a 128^2 float64 grid has 16 tiles of 8 columns for
// 152 SMs and 128 of one (step 96 -> 39 us with the x passes split the same
// way), a 384 x 192 float32 one 24 and 192 (57 -> 26 us). f(width constant, args with the tiling, blocks).
template <typename Real, int N, int VAR, typename F>
static cudaError_t col_pick(const ColArgs& a0, int runs, F&& f) {
  typedef ColShape<Real, N, VAR> W;
  constexpr int CW = W::CW;
  constexpr bool TWO = W::TWO;
  ColArgs a = a0;
  long long blocks = col_tiles(a, CW * W::wide(), TWO);
  if (blocks * runs >= kSMs || W::narrow() == W::wide()) return f(std::integral_constant<int, W::wide()>(), a, blocks);
  if constexpr (W::mid() != W::wide()) {
    a = a0;
    blocks = col_tiles(a, CW * W::mid(), TWO);
    if (blocks * runs >= kSMs) return f(std::integral_constant<int, W::mid()>(), a, blocks);
  }
  a = a0;
  blocks = col_tiles(a, CW * W::narrow(), TWO);
  return f(std::integral_constant<int, W::narrow()>(), a, blocks);
}

// One variant of the column pass at every length.
template <typename Real, int VAR>
cudaError_t launch_col_var(int n, const ColArgs& a, const MulArgs& m, const void* tw, cudaStream_t st) {
  switch (n) {
#define FSE_CASE(n)                                                                                          \
  case n:                                                                                                    \
    return col_pick<Real, n, VAR>(a, 1, [&](auto w, const ColArgs& at, long long blocks) {                   \
      return col_launch<Real, n, VAR, decltype(w)::value>(at, m, blocks, tw, st);                            \
    });
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

template <typename Real, int NX, int LN, int KIND>
static cudaError_t x_launch(const XArgs& a, const void* twn, const void* tw2n, cudaStream_t st) {
  typedef XLaunch<Real, NX, LN, KIND> K;
  typedef typename TwOf<Real>::T C;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_xpass<Real, NX, LN, KIND>, K::smem(), done);
  if (e != cudaSuccess) return e;
  const int blocks = (a.nlines + LN - 1) / LN;
  if (blocks <= 0) return cudaSuccess;
  XArgs af = a;
  fill_f32(af);
  return launch_pass(k_xpass<Real, NX, LN, KIND>, (unsigned)blocks, K::threads, K::smem(), st, af,
                     reinterpret_cast<const C*>(twn), reinterpret_cast<const C*>(tw2n));
}

// One kind of x pass at every length.
template <typename Real, int KIND>
cudaError_t launch_xpass(int nx, const XArgs& a, const void* twn, const void* tw2n, cudaStream_t st) {
  switch (nx) {
#define FSE_CASE(n)                                                                              \
  case n:                                                                                        \
    return xpass_pick<Real, n>(a.nlines, 1) == XWidths<Real, n>::wide()                          \
               ? x_launch<Real, n, XWidths<Real, n>::wide(), KIND>(a, twn, tw2n, st)             \
               : x_launch<Real, n, XWidths<Real, n>::narrow(), KIND>(a, twn, tw2n, st);
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

template <typename Real> int xpass_tiles(int nx, int nlines) {
  switch (nx) {
#define FSE_CASE(n) \
  case n:           \
    return (nlines + xpass_pick<Real, n>(nlines, 1) - 1) / xpass_pick<Real, n>(nlines, 1);
    FSE_SIZES(FSE_CASE)
#undef FSE_CASE
    default:
      return 0;
  }
}

}  // namespace fse
