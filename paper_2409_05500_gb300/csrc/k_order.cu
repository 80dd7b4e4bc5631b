// Algorithm 1: the accelerated causal-order search over the static
// precomputed matrix.  For k = 1..m the candidate c_k in U minimising
//     M_i = sum_{j in U, j != i} min(0, D_ij)^2            (Eq. 3)
// is appended to the order and removed from U (ties: lowest index).
//
// GB300 design.  The m steps are strictly sequential, so the search is one
// CTA and its cost is latency per step.  FP64 issues at 1/64 of the FP32 rate
// on this part, so the running sums S_i = M_i are kept as double-float pairs
// (hi + lo, two FP32 numbers, ~48-bit significand) and updated with TwoSum
// after each pick, S_i -= P_{i,c}.  The argmin compares an order-preserving
// 64-bit integer key built from (hi, lo) and the index, so no floating-point
// compare sits on the critical path; scores closer than about 2^-35 relative
// are taken as tied and go by index (order_search.cuh).
// The initial sums are computed in FP64 by a parallel kernel; the per-step
// relative gaps are computed after the search by another.  Subtracting the
// removed column instead of re-summing over U gives the same sums as the
// literal recomputation up to rounding (~1e-14 relative).
#include <algorithm>
#include <mutex>

#include "order_search.cuh"


namespace vl {

namespace {

using namespace search;
static_assert(VL_MAX_M <= 16 * STH, "ordering holds at most sixteen variables per thread");
static_assert(VL_MAX_M <= 4096, "the search key holds the variable index in 12 bits");

// Pt[c * m + i] = min(0, D[i * m + c])^2 as a double-float pair.
__global__ void pt_kernel(const double* __restrict__ D, int m, float2* __restrict__ pt, int* st) {
  pdl_begin(D, pt, st);
  __shared__ double tile[32][33];
  const int c0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int r = ty; r < 32; r += 8) {
    int i = i0 + r, c = c0 + tx;
    double v = 0.0;
    if (i < m && c < m) {
      double d = D[(int64_t)i * m + c];
      if (!isfinite(d)) set_status(st, VL_ERR_NONFINITE);
      v = (i != c && d < 0.0) ? d * d : 0.0;
    }
    tile[r][tx] = v;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    int c = c0 + r, i = i0 + tx;
    if (c < m && i < m) {
      double v = tile[tx][r];
      float hi = (float)v;
      pt[(int64_t)c * m + i] = make_float2(hi, (float)(v - (double)hi));
    }
  }
}

// S_i = sum_{j != i} min(0, D_ij)^2 in FP64, one warp per row, fixed order.
__global__ void rowsum_kernel(const double* __restrict__ D, int m, float* __restrict__ sh,
                              float* __restrict__ sl) {
  pdl_begin(D, sh, sl);
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= m) return;
  double s = 0.0;
  for (int j = lane; j < m; j += 32) {
    double d = D[(int64_t)i * m + j];
    if (j != i && d < 0.0) s += d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    float hi = (float)s;
    sh[i] = hi;
    sl[i] = (float)(s - (double)hi);
  }
}

// This thread's variables at the start of the search.
template <int PER, int NW>
__device__ __forceinline__ void load_scores(const float* __restrict__ sh0,
                                            const float* __restrict__ sl0, int m,
                                            float (&hi)[PER], float (&lo)[PER],
                                            bool (&alive)[PER]) {
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int i = threadIdx.x + q * 32 * NW;
    alive[q] = i < m;
    hi[q] = alive[q] ? sh0[i] : 0.f;
    lo[q] = alive[q] ? sl0[i] : 0.f;
  }
}

// Where P_{i,c} comes from decides a step's latency (measured dependent loads:
// L2 300 to 530 clocks, distributed shared memory 290, a CTA's own shared
// memory 33, L1 38), and m decides what fits:
//   m <= 160        P in the CTA's own shared memory (order_local_kernel),
//   160 < m <= 448  in the shared memory of a cluster (order_cluster_kernel),
//   beyond          in L2, with the columns of likely picks fetched into L1
//                   ahead of time (order_kernel).
// Measured, whole call without gaps, against a search with one variable per
// thread, a branch around every dead variable, P in L2 below m = 64 and beyond
// 448 (no fetching ahead) and in a cluster between: m = 32 27 -> 17 us, 64
// 37 -> 22, 100 52 -> 29, 160 74 -> 41, 256 107 -> 78, 400 165 -> 133, 800
// 561 -> 371, 1600 1444 -> 1108; in a later run 1600 1597 -> 1141, 2048 2281 -> 1468,
// 3000 4883 -> 3412, 4096 7758 -> 4733 (256 threads with up to 16 variables each, where
// 1024 had up to 4).

// Search with P in global memory: Pt[c * m + i] = P_{i,c}.  The eventual pick
// is usually some warp's minimum for a few steps before it wins (in 60 to 80 %
// of the steps, on measured D), so each warp, when its minimum changes, brings
// that variable's column into L1: one asynchronous four-byte copy per line, to
// a word nobody reads (prefetch.global.L1 leaves L1 untouched on this part, and
// a plain load's destination register made later steps wait for it).
template <int PER>
__global__ void __launch_bounds__(STH) order_kernel(const float2* __restrict__ pt,
                                                    const float* __restrict__ sh0,
                                                    const float* __restrict__ sl0, int m,
                                                    int32_t* __restrict__ order,
                                                    float2* __restrict__ spick) {
  float hi[PER], lo[PER];
  bool alive[PER];
  load_scores<PER, SW>(sh0, sl0, m, hi, lo, alive);
  __shared__ uint32_t sinks[STH];
  const uint32_t sink = (uint32_t)__cvta_generic_to_shared(&sinks[threadIdx.x]);
  int last = -1;
  search_steps<PER, SW>(
      hi, lo, alive, m, 0, -1, order, spick,
      [&](int c, int q) {
        return __ldg(pt + (int64_t)c * m + min((int)threadIdx.x + q * STH, m - 1));
      },
      [&](int j) {
        if (j == last || j >= m) return;
        last = j;
        const char* col = reinterpret_cast<const char*>(pt + (int64_t)j * m);
        for (int o = (threadIdx.x & 31) * 128; o < 8 * m; o += 32 * 128)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sink), "l"(col + o));
      });
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// Copy cnt columns' rows i0 .. i0 + R - 1 of P into sm[c R + il] (zeros beyond
// m), eight loads in flight per thread.
__device__ __forceinline__ void stage_rows(const float2* __restrict__ pt, int m, int i0, int R,
                                           float2* sm) {
  const int tot = R * m;
  for (int b = threadIdx.x; b < tot; b += 8 * blockDim.x) {
    float2 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int idx = b + u * blockDim.x;
      const int c = idx / R, i = i0 + idx - c * R;
      v[u] = idx < tot && i < m ? __ldg(pt + (int64_t)c * m + i) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int idx = b + u * blockDim.x;
      if (idx < tot) sm[idx] = v[u];
    }
  }
}

constexpr int OL_MAX_M = 160;  // 8 m^2 bytes fit one CTA's shared memory
constexpr int OC_TH = 512;     // threads that stage P (the first 32 NW of them search)

// The search with all of P in this CTA's shared memory, one variable per thread.
template <int NW>
__global__ void __launch_bounds__(OC_TH) order_local_kernel(const float2* __restrict__ pt,
                                                            const float* __restrict__ sh0,
                                                            const float* __restrict__ sl0, int m,
                                                            int32_t* __restrict__ order,
                                                            float2* __restrict__ spick) {
  pdl_wait(pt, sh0, sl0, order, spick);
  extern __shared__ __align__(16) float2 oc_rows[];
  stage_rows(pt, m, 0, m, oc_rows);
  __syncthreads();
  if (threadIdx.x >= 32 * NW) return;
  float hi[1], lo[1];
  bool alive[1];
  load_scores<1, NW>(sh0, sl0, m, hi, lo, alive);
  const int i = min((int)threadIdx.x, m - 1);
  search_steps<1, NW>(
      hi, lo, alive, m, 0, -1, order, spick, [&](int c, int) { return oc_rows[c * m + i]; },
      NoAhead());
}

// The same search with P held in distributed shared memory: a cluster of
// OC_CTAS CTAs, CTA t keeping the rows i in [t R, (t+1) R) of P for every
// column c (R = ceil(m / OC_CTAS), layout [c][i - t R] as (hi, lo) pairs).  CTA 0
// runs the search; the others only hold their rows until it is done.  The only
// synchronisation is a cluster barrier after the rows are loaded and one at the
// end, so no CTA leaves while its rows can still be read.
constexpr int OC_CTAS = 8;
constexpr int OC_MAX_M = 448;  // R m (hi, lo) pairs must fit one CTA's shared memory

inline size_t oc_smem(int m) {
  const int R = (m + OC_CTAS - 1) / OC_CTAS;
  return (size_t)R * m * sizeof(float2);
}

template <int NW>
__global__ void __launch_bounds__(OC_TH) order_cluster_kernel(const float2* __restrict__ pt,
                                                              const float* __restrict__ sh0,
                                                              const float* __restrict__ sl0, int m,
                                                              int32_t* __restrict__ order,
                                                              float2* __restrict__ spick) {
  pdl_wait(pt, sh0, sl0, order, spick);
  extern __shared__ __align__(16) float2 oc_rows[];
  unsigned rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int R = (m + OC_CTAS - 1) / OC_CTAS;
  stage_rows(pt, m, (int)rank * R, R, oc_rows);
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (rank == 0 && threadIdx.x < 32 * NW) {
    float hi[1], lo[1];
    bool alive[1];
    load_scores<1, NW>(sh0, sl0, m, hi, lo, alive);
    // this thread's row: owner CTA and local index, as a shared::cluster base
    const int i = min((int)threadIdx.x, m - 1), own = i / R;
    uint32_t base = (uint32_t)__cvta_generic_to_shared(oc_rows) + 8u * (uint32_t)(i - own * R);
    asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(base) : "r"(own));
    const uint32_t stride = 8u * (uint32_t)R;
    search_steps<1, NW>(
        hi, lo, alive, m, 0, -1, order, spick,
        [&](int c, int) {
          float2 v;
          asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];"
                       : "=f"(v.x), "=f"(v.y)
                       : "r"(base + stride * (uint32_t)c)
                       : "memory");
          return v;
        },
        NoAhead());
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Launch the cluster search; false if the cluster cannot be launched (the
// caller then runs order_kernel).
template <int NW>
bool launch_order_cluster(const OrderWs& w, int m, int32_t* order, float2* spick,
                          Lane s) {
  static SmemOptIn smem;
  if (!smem.allow(order_cluster_kernel<NW>, oc_smem(OC_MAX_M))) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(OC_CTAS, 1, 1);
  cfg.blockDim = dim3(OC_TH, 1, 1);
  cfg.dynamicSmemBytes = oc_smem(m);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = OC_CTAS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  at[1] = pdl_attribute();
  cfg.numAttrs = s.overlap ? 2 : 1;
  note_launch();
  if (cudaLaunchKernelEx(&cfg, order_cluster_kernel<NW>, (const float2*)w.pt,
                         (const float*)w.sh, (const float*)w.sl, m, order, spick) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

// Launch the search in one CTA's shared memory; false as above.
template <int NW>
bool launch_order_local(const OrderWs& w, int m, int32_t* order, float2* spick, Lane s) {
  static SmemOptIn smem;
  if (!smem.allow(order_local_kernel<NW>, OL_MAX_M * OL_MAX_M * sizeof(float2))) return false;
  if (launch(order_local_kernel<NW>, 1, OC_TH, (size_t)m * m * sizeof(float2), s, w.pt, w.sh, w.sl,
             m, order, spick) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

// Gaps after the search, from the order: variable i replays its score S_i =
// sum_{j in U} P_ij step by step in FP64; at the step that picks it, it records
// its score as the minimum s1[k]; at earlier steps it offers its score to the
// step's runner-up s2[k] (atomic minimum of an ordered key).  The replay is a
// serial chain of FP64 subtractions per variable (about 40 clocks each), so
// everything else is kept off it: a CTA takes GAP_V variables and GAP_T steps at
// a time, all threads load and convert the tile's P (FP64 conversions issue at
// 1.6 per clock per SM: few variables per CTA spread them over the SMs), one
// warp runs the chains, and one thread per step reduces the GAP_V scores to one
// atomic.  The gaps of m = 800 add 62 to 70 us (290 to 310 with one thread doing all
// of it for each variable).
constexpr int GAP_V = 8, GAP_T = 64, GAP_TH = 128;
__global__ void __launch_bounds__(GAP_TH)
    gap_scores_kernel(const float2* __restrict__ pt, const float* __restrict__ sh0,
                      const float* __restrict__ sl0, const int32_t* __restrict__ order, int m,
                      double* __restrict__ s1, unsigned long long* __restrict__ s2) {
  pdl_begin(pt, sh0, sl0, order, s1, s2);
  constexpr int PER = GAP_V * GAP_T / GAP_TH;
  __shared__ double ps[GAP_T][GAP_V];  // P_i,order[k], then the scores before step k
  __shared__ int pos[GAP_V];           // the step of i's own pick, once reached
  const int tid = threadIdx.x, v = tid % GAP_V, i0 = blockIdx.x * GAP_V;
  const int i = min(i0 + v, m - 1);
  if (tid < GAP_V) pos[tid] = i0 + tid < m ? m : -1;
  double s = (double)sh0[i] + (double)sl0[i];
  float2 p[PER];  // the next tile's entries of steps t = tid / GAP_V + q GAP_TH / GAP_V
  int c[PER];
  auto load = [&](int t0) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int k = t0 + tid / GAP_V + q * (GAP_TH / GAP_V);
      c[q] = k < m ? order[k] : -1;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q)
      p[q] = c[q] >= 0 ? pt[(int64_t)c[q] * m + i] : make_float2(0.f, 0.f);
  };
  load(0);
  __syncthreads();
  for (int t0 = 0; t0 < m; t0 += GAP_T) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int t = tid / GAP_V + q * (GAP_TH / GAP_V);
      ps[t][v] = (double)p[q].x + (double)p[q].y;
      if (c[q] == i0 + v) pos[v] = t0 + t;
    }
    __syncthreads();
    if (t0 + GAP_T < m) load(t0 + GAP_T);
    if (tid < GAP_V) {
#pragma unroll 8
      for (int t = 0; t < GAP_T; ++t) {
        const double x = ps[t][v];
        ps[t][v] = s;
        s -= x;
      }
    }
    __syncthreads();
    const int k = t0 + tid;
    bool more = false;
    if (tid < GAP_T && k < m) {
      unsigned long long best = ~0ull;
#pragma unroll
      for (int u = 0; u < GAP_V; ++u) {
        const double x = ps[tid][u];
        if (k == pos[u]) s1[k] = x;
        if (k < pos[u]) {
          const unsigned long long key = dkey(x);
          best = key < best ? key : best;
        }
      }
      if (best != ~0ull) {
        atomicMin(&s2[k], best);
        more = true;  // a later step may still see one of these variables
      }
    }
    if (!__syncthreads_or(more)) break;
  }
}

__global__ void gap_kernel(const double* __restrict__ s1, const unsigned long long* __restrict__ s2,
                           int m, double* __restrict__ gap) {
  pdl_begin(s1, s2, gap);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  if (s2[k] == ~0ull) {
    gap[k] = __longlong_as_double(0x7ff0000000000000LL);
    return;
  }
  const double a = s1[k], b = dkey_inv(s2[k]);
  const double den = fmax(fmax(fabs(a), fabs(b)), 1e-300);
  gap[k] = (b - a) / den;
}

}  // namespace

OrderWs order_ws_layout(void* ws, int m) {
  OrderWs w;
  char* p = static_cast<char*>(ws);
  w.pt = reinterpret_cast<float2*>(p);
  w.sh = reinterpret_cast<float*>(w.pt + (size_t)m * m);
  w.sl = w.sh + m;
  w.s1 = reinterpret_cast<double*>(((uintptr_t)(w.sl + m) + 15) & ~(uintptr_t)15);
  w.s2 = reinterpret_cast<unsigned long long*>(w.s1 + m);
  return w;
}

void launch_order_gaps(void* ws, int m, const int32_t* order, double* gap,
                       Lane s) {
  const OrderWs w = order_ws_layout(ws, m);
  cudaMemsetAsync(w.s2, 0xff, (size_t)m * sizeof(unsigned long long), s);
  launch(gap_scores_kernel, (m + GAP_V - 1) / GAP_V, GAP_TH, 0, s, w.pt, w.sh, w.sl, order, m,
         w.s1, w.s2);
  launch(gap_kernel, (m + 255) / 256, 256, 0, s, w.s1, w.s2, m, gap);
}

size_t order_ws_bytes(int m) {
  return (size_t)m * m * 2 * sizeof(float) + (size_t)m * 2 * sizeof(float) +
         (size_t)m * sizeof(float4) + 1024;
}

bool launch_causal_order(const double* D, int m, void* ws, int32_t* order, double* gap, int* st,
                         Lane s, float2* spick) {
  const OrderWs w = order_ws_layout(ws, m);
  dim3 grid((m + 31) / 32, (m + 31) / 32), block(32, 8);
  launch(pt_kernel, grid, block, 0, s, D, m, w.pt, st);
  launch(rowsum_kernel, (m + 7) / 8, 256, 0, s, D, m, w.sh, w.sl);
  bool done = false;
  if (m <= 32)
    done = launch_order_local<1>(w, m, order, spick, s);
  else if (m <= 64)
    done = launch_order_local<2>(w, m, order, spick, s);
  else if (m <= 128)
    done = launch_order_local<4>(w, m, order, spick, s);
  else if (m <= OL_MAX_M)
    done = launch_order_local<8>(w, m, order, spick, s);
  else if (m <= 256)
    done = launch_order_cluster<8>(w, m, order, spick, s);
  else if (m <= OC_MAX_M)
    done = launch_order_cluster<16>(w, m, order, spick, s);
  if (!done) {
    const Lane alone(s, false);  // order_kernel has no pdl_wait: 1.5 us of 250 or more
    const auto search = m <= 2 * STH   ? order_kernel<2>
                        : m <= 4 * STH ? order_kernel<4>
                        : m <= 8 * STH ? order_kernel<8>
                                       : order_kernel<16>;
    if (launch(search, 1, STH, 0, alone, w.pt, w.sh, w.sl, m, order, spick) != cudaSuccess)
      return false;
  }
  if (gap) launch_order_gaps(ws, m, order, gap, s);
  return true;
}

}  // namespace vl

// ------------------------------------------------------------------------
// Allocation-free variant of the search, for callers that must not allocate
// device memory after start-up.  Its scratch is this file-scope array; every
// GPU that loads the library holds it until the process exits.
namespace vl {
namespace {

constexpr size_t kNoallocBytes =
    (size_t)VL_NOALLOC_MAX_M * VL_NOALLOC_MAX_M * 2 * sizeof(float) +
    (size_t)VL_NOALLOC_MAX_M * 2 * sizeof(float) + (size_t)VL_NOALLOC_MAX_M * sizeof(float4) +
    1024;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

constexpr int kMaxDevices = 64;
void* g_noalloc_ptr[kMaxDevices] = {};
std::mutex g_noalloc_mutex;

}  // namespace

}  // namespace vl

extern "C" vl_status vl_causal_order_noalloc(void* cuda_stream, const double* D, int m,
                                             int32_t* order, double* gap) {
  using namespace vl;
  if (!D || !order) return VL_ERR_ARG;
  if (m < 1) return VL_ERR_SHAPE;
  if (m > VL_NOALLOC_MAX_M) return VL_ERR_UNSUPPORTED;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return VL_ERR_CUDA;
  }
  void* scratch;
  {
    // first call on this device: resolve the array's device address (host
    // code cannot use the symbol itself: on the host it names a stand-in)
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      void* ptr = nullptr;
      if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
        cudaGetLastError();
        return VL_ERR_CUDA;
      }
      g_noalloc_ptr[dev] = ptr;
    }
    scratch = g_noalloc_ptr[dev];
  }
  if (order_ws_bytes(m) > kNoallocBytes) return VL_ERR_UNSUPPORTED;
  // an error the caller left pending is not this call's: report only an
  // error that the launches below raise (and clear only that one)
  const cudaError_t before = cudaPeekAtLastError();
  const bool launched = launch_causal_order(D, m, scratch, order, gap, nullptr,
                                            Lane(static_cast<cudaStream_t>(cuda_stream)));
  const cudaError_t after = cudaPeekAtLastError();
  if (launched && (after == cudaSuccess || after == before)) return VL_OK;
  cudaGetLastError();
  return VL_ERR_CUDA;
}
