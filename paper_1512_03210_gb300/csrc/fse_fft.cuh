// fse_fft.cuh -- complex scalars, asynchronous copies and unit-modulus products shared by the passes.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fse {

template <typename R> struct Cplx;
template <> struct Cplx<float> { typedef float2 T; };
template <> struct Cplx<double> { typedef double2 T; };

__device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }

// Asynchronous 4/8/16-byte global -> shared copy (cp.async, completes in the
// background) and the wait for all of a thread's outstanding copies.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
  static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async size");
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  if constexpr (BYTES == 16)  // 16-byte copies bypass L1 (.cg): the data is streamed once
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// Bulk prefetch of a contiguous global range into L2 (address and size
// multiples of 16 bytes); no completion to wait for.
__device__ __forceinline__ void prefetch_l2_bulk(const void* gmem, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(gmem), "r"(bytes) : "memory");
}

// Error of the modulus of a float pair, c^2 + s^2 - 1, computed exactly enough
// to correct it: the two squares are split into rounded product plus fma
// remainder, and the larger square minus one is exact (Sterbenz).
__device__ __forceinline__ float norm_err(float c, float s) {
  const bool big = fabsf(c) >= fabsf(s);
  const float a = big ? c : s, b = big ? s : c;
  const float pa = a * a, ea = fmaf(a, a, -pa);
  const float pb = b * b, eb = fmaf(b, b, -pb);
  return ((pa - 1.0f) + pb) + (ea + eb);
}

// v times the float pair (c, s) of a unit-modulus factor, with the pair's
// modulus error folded into the products before their final rounding (the
// factor's remainder is taken as -(|w|^2 - 1)/2 w from norm_err).
__device__ __forceinline__ float2 unit_mul(float2 v, float c, float s, bool conj_w) {
  const float h = -0.5f * norm_err(c, s);
  const float lc = h * c, ls = conj_w ? -h * s : h * s;
  const float sc = conj_w ? -s : s;
  const float lr = v.x * lc - v.y * ls, li = v.x * ls + v.y * lc;
  return make_float2(fmaf(v.x, c, fmaf(-v.y, sc, lr)), fmaf(v.x, sc, fmaf(v.y, c, li)));
}
__device__ __forceinline__ double2 unit_mul(double2 v, double c, double s, bool conj_w) {
  const double sc = conj_w ? -s : s;
  return make_double2(v.x * c - v.y * sc, v.x * sc + v.y * c);
}

// Deterministic float64 block sum (blockDim.x <= 1024; the last warp may be
// partly filled); result in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  const int lanes = min(32, (int)blockDim.x - 32 * w);
  const unsigned mask = lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u;
  for (int o = 16; o > 0; o >>= 1) {
    const double t = __shfl_down_sync(mask, v, o);
    if (l + o < lanes) v += t;
  }
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  v = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < nw; ++i) v += sh[i];
  return v;
}

// Deterministic float64 block sums of K values; sh holds K * blockDim.x
// doubles. Warp w sums values w, w + nw, ... over the block (a float64 warp
// instruction holds its scheduler for 64 cycles whatever lanes it has, so the
// additions are packed into few full warps). out(k, sum) is called by one thread.
template <int K, typename F> __device__ __forceinline__ void block_sums(const double (&s)[K], double* sh, F&& out) {
  const int n = blockDim.x, w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = n >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) sh[k * n + threadIdx.x] = s[k];
  __syncthreads();
  if (w >= nw) return;  // a partly filled last warp does not take part
  for (int k = w; k < K; k += nw) {
    double v = 0.0;
    for (int i = l; i < n; i += 32) v += sh[k * n + i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (l == 0) out(k, v);
  }
}

}  // namespace fse
