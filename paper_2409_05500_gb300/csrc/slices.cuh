// The exact-slice split of the tensor-core products (k_tcgram.cu) and block
// reductions, shared by the kernels that prepare their operands.
#pragma once

#include <cuda_bf16.h>

#include "vl_internal.cuh"

namespace vl {

// Exponent e with max < 2^e from the bits of a non-negative double (0 -> 0),
// clamped so that the FP32 scale 2^(7 - e) is finite and normal (rows whose
// largest entry is below 2^-100 are treated as zero-ish; the mixed path
// takes no entries above 2^120).
__device__ __forceinline__ int clamp_exp(int e) { return min(120, max(-100, e)); }
__device__ __forceinline__ int exp_above(unsigned long long bits) {
  if (bits == 0) return 0;
  return clamp_exp((int)((bits >> 52) & 0x7ff) - 1022);
}

// Three integer slices of y in (-128, 128) given as an FP32 pair (yh + yl).
__device__ __forceinline__ void slice3(float yh, float yl, __nv_bfloat16& s0, __nv_bfloat16& s1,
                                       __nv_bfloat16& s2) {
  const float a0 = rintf(yh);
  const float r1 = ((yh - a0) + yl) * 256.f;
  const float a1 = rintf(r1);
  const float a2 = rintf((r1 - a1) * 256.f);
  s0 = __float2bfloat16_rn(a0);
  s1 = __float2bfloat16_rn(a1);
  s2 = __float2bfloat16_rn(a2);
}

__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long v,
                                                            unsigned long long* red) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long b = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) b = red[q] > b ? red[q] : b;
    red[0] = b;
  }
  __syncthreads();
  return red[0];
}

// Sums over the block (64 to 256 threads, a power of two) in FP64, in every
// thread.  An FP64 instruction keeps a scheduler's FP64 unit for 64 clocks, so it
// is their number that counts.  block_sum adds in the order of a shuffle tree in
// each warp and one over the warps' sums, of which only the sums that go on are
// formed: three levels folded through shared memory, the rest by the first warp.
// (Where a mean decides how a sample rounds to FP32, its order stays fixed: an ulp
// of it moves a coefficient by an ulp of FP32 now and then.)  block_fold and
// block_sum2 (two sums, the second's last warp beside the first's) halve the block
// instead, 0.5 us a sum faster.  red: 2 blockDim.x doubles.  f is applied to the
// sum by one thread (a division or root there costs one warp 600 to 1,000 clocks,
// not every warp).
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <class F>
__device__ __forceinline__ double block_sum(double v, double* red, F f) {
  const int tid = threadIdx.x, n = blockDim.x;
  double* r2 = red + n;
  __syncthreads();
  red[tid] = v;
  __syncthreads();
  // value (w, l) at w 2h + l: (w, l) + (w, l + h) goes to w h + l
  if (tid < n / 2) r2[tid] = red[2 * tid - (tid & 15)] + red[2 * tid - (tid & 15) + 16];
  __syncthreads();
  if (tid < n / 4) red[tid] = r2[2 * tid - (tid & 7)] + r2[2 * tid - (tid & 7) + 8];
  __syncthreads();
  if (tid < 32) {
    v = tid < n / 8 ? red[2 * tid - (tid & 3)] + red[2 * tid - (tid & 3) + 4] : 0.0;
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    for (int o = 16; o >= 4; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (tid == 0) r2[0] = f(v);
  }
  __syncthreads();
  return r2[0];
}
template <class F>
__device__ __forceinline__ double block_fold(double v, double* red, F f) {
  const int tid = threadIdx.x;
  __syncthreads();
  red[tid] = v;
  __syncthreads();
  for (int h = blockDim.x >> 1; h >= 32; h >>= 1) {
    if (tid < h) red[tid] = v = v + red[tid + h];
    __syncthreads();
  }
  if (tid < 32) {
    v = warp_sum_f64(v);
    if (tid == 0) red[0] = f(v);
  }
  __syncthreads();
  return red[0];
}
// t / n, correctly rounded, from inv = 1 / n correctly rounded (Markstein 1990: a
// quotient within an ulp, its exact remainder, one correction): three instructions
// inline for a call into the division of 600 clocks and its instruction fetches.
__device__ __forceinline__ double div_by(double t, int n, double inv) {
  const double q = t * inv;
  return fma(fma(-q, (double)n, t), inv, q);
}
__device__ __forceinline__ double block_sum(double v, double* red) {
  return block_sum(v, red, [](double t) { return t; });
}
__device__ __forceinline__ void block_sum2(double& a, double& b, double* red) {
  const int tid = threadIdx.x, n = blockDim.x;
  double* rb = red + n;
  __syncthreads();
  red[tid] = a;
  rb[tid] = b;
  __syncthreads();
  // the lower half of the threads folds a, the upper half b
  const bool lo = tid < n / 2;
  double* r = lo ? red : rb;
  const int t = lo ? tid : tid - n / 2;
  double v = r[t] + r[t + n / 2];
  for (int h = n >> 2; h >= 32; h >>= 1) {
    r[t] = v;
    __syncthreads();
    if (t < h) v += r[t + h];
  }
  if (t < 32) {
    v = warp_sum_f64(v);
    if (t == 0) r[0] = v;
  }
  __syncthreads();
  a = red[0];
  b = rb[0];
}

__device__ __forceinline__ bool is_finite(double v) {
  return ((uint32_t)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

}  // namespace vl
