// Device pieces of Algorithm 1's search (Eq. 3 argmin over the remaining
// set), shared by the plain search (k_order.cu) and the search resumed after
// an FP64 re-evaluation of a near tie (k_certify.cu).
//
// The running sums S_i = sum_{j in U, j != i} min(0, D_ij)^2 are double-float
// pairs (hi + lo, two FP32 numbers, ~48-bit significand) updated with TwoSum,
// because FP64 issues at 1/64 of the FP32 rate on this part.  The argmin
// compares an order-preserving 64-bit integer key built from (hi, lo) and the
// index.
#pragma once

#include "vl_internal.cuh"

namespace vl {
namespace search {

constexpr int SW = 8;           // warps of a search with several variables per thread
constexpr int STH = 32 * SW;    // and its threads
constexpr int SW_MAX = 16;      // most warps that search

// order-preserving map float -> uint32 (valid for every non-NaN value)
__device__ __forceinline__ uint32_t fkey(float f) {
  uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// (hi, lo) -= (ph, pl) in double-float, renormalised so |lo| <= ulp(hi)/2
// (then the pair order equals the order of (key(hi), key(lo))).
__device__ __forceinline__ void df_sub(float& hi, float& lo, float ph, float pl) {
  float s = hi - ph;
  float bp = s - hi;
  float err = (hi - (s - bp)) + (-ph - bp);
  float l = lo - pl + err;
  float h2 = s + l;
  lo = l - (h2 - s);
  hi = h2;
}

// Search key of a live variable: (fkey(hi), fkey(lo) with its low 12 bits
// replaced by the index).  Compared as a 64-bit integer it orders by the
// double-float score and then by index; dropping 12 bits of lo merges
// scores closer than about 2^-35 relative into index order, far below any
// gap the method distinguishes.  A dead variable is (~0, ~0).
// The score a key encodes (lo without its 12 index bits), as a pair.
__device__ __forceinline__ float2 skey_pair(uint2 k) {
  return make_float2(fkey_inv(k.x), fkey_inv(k.y & 0xfffff000u));
}
// warp-wide minimum key, in every lane
__device__ __forceinline__ uint2 warp_kmin(uint2 k) {
  const uint32_t full = 0xffffffffu;
  const uint32_t h = __reduce_min_sync(full, k.x);
  const uint32_t l = __reduce_min_sync(full, k.x == h ? k.y : 0xffffffffu);
  return make_uint2(h, l);
}

// order-preserving map double -> uint64
__device__ __forceinline__ unsigned long long dkey(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double dkey_inv(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
  return __longlong_as_double((long long)b);
}

struct NoAhead {
  __device__ __forceinline__ void operator()(int) const {}
};

// Steps kbeg .. m-1 of the search by the first NW warps of a CTA (NW = 1, 2, 4,
// 8 or 16; a named barrier, so the CTA may hold more), each thread owning PER
// variables (i = tid + q 32 NW).  A step is one latency chain: keys (the
// smallest high word over the thread and the warp first, then the low words
// that go with it), the warp's minimum to a shared slot of the step's parity,
// one barrier, the minimum over the NW slots (in every warp), the fetch of P's
// column, S_i -= P_{i,c}.  No branch depends on a variable: dead ones compute
// along, so that every warp takes the same straight path.  No second barrier:
// slots alternate by parity and a warp can run at most one step ahead of the
// slowest.  forced >= 0 makes step kbeg pick that variable without a search
// (its score is then not recorded).  spick (optional): the winning score of
// every searched step, as a pair.  fetch(c, q) loads P_{i,c} as a pair for the
// thread's variable q (any valid address for i >= m); ahead(j), called by every
// warp while the fetch is in flight, names the warp's own candidate, a likely
// later pick.
template <int PER, int NW, class Fetch, class Ahead>
__device__ __forceinline__ void search_steps(float (&hi)[PER], float (&lo)[PER],
                                             bool (&alive)[PER], int m, int kbeg, int forced,
                                             int32_t* __restrict__ order,
                                             float2* __restrict__ spick, Fetch fetch,
                                             Ahead ahead) {
  __shared__ uint2 wb[2][SW_MAX];
  constexpr int nthr = 32 * NW;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // a live variable's high key is below ~0 (only a NaN's can reach it)
  uint32_t dead[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) dead[q] = alive[q] ? 0u : 0xffffffffu;
  for (int k = kbeg; k < m; ++k) {
    int c = forced, own = -1;
    if (k != kbeg || forced < 0) {
      uint32_t hk[PER], bh = 0xffffffffu, bl = 0xffffffffu;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        hk[q] = fkey(hi[q]) | dead[q];
        bh = min(bh, hk[q]);
      }
      bh = __reduce_min_sync(0xffffffffu, bh);
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const uint32_t lk =
            ((fkey(lo[q]) & 0xfffff000u) | (uint32_t)(threadIdx.x + q * nthr)) | dead[q];
        bl = min(bl, hk[q] == bh ? lk : 0xffffffffu);
      }
      bl = __reduce_min_sync(0xffffffffu, bl);
      uint2 g = make_uint2(bh, bl);
      own = (int)(bl & 0xfffu);
      if constexpr (NW > 1) {
        const int ph = k & 1;
        if (lane == 0) wb[ph][wid] = g;
        asm volatile("bar.sync 1, %0;" ::"n"(nthr) : "memory");
        g = warp_kmin(wb[ph][lane & (NW - 1)]);
      }
      c = (int)(g.y & 0xfffu);
      if (spick && threadIdx.x == 0) spick[k] = skey_pair(g);
    }
    float2 p[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) p[q] = fetch(c, q);
    if (threadIdx.x == 0) order[k] = c;
    ahead(own);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      df_sub(hi[q], lo[q], p[q].x, p[q].y);
      if ((int)threadIdx.x + q * nthr == c) dead[q] = 0xffffffffu;
    }
  }
}

}  // namespace search
}  // namespace vl
