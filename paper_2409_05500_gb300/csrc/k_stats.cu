// Per-variable statistics and data layout kernels.
//
//  * prep_lags    : mixed path of the VAR (Sec. 4.1): full-series mean of each
//                   variable, the centred FP32 copy, the mean of every lag
//                   window (the VAR intercept is equivalent to centring each
//                   window) and the bf16 slices of the windows.
//  * var_prep     : the same statistics and the centred copy on the FP64 path.
//  * measure_prep : mixed path of the measure: mean and 1/std (population) of
//                   each variable (Sec. 3 step 1), its entropy H(x_i) (Sec. 4.2
//                   item 1 precomputes it once), the bf16 slices of the centred
//                   row and the standardized row.
//  * standardize  : mean, 1/std and entropy on the FP64 path.
//  * transpose_std: standardized residuals, time-major, zero padded, in the
//                   layout the pairwise kernel stages into shared memory.
//
// All of them are bound by the number of FP64 instructions (1.6 per clock per SM,
// conversions included): a row is read in as few passes as its statistics allow,
// scalar divisions and roots are taken by one thread, conversions run on the
// integer pipe.  m = 400, n = 2500: prep_lags 26 us (28 + 11 as two kernels with a
// pass per window), measure_prep 33 us (33 + 19 as two).
#include <cmath>

#include "fp64_bits.cuh"
#include "fx64.cuh"
#include "slices.cuh"
#include "vl_internal.cuh"

namespace vl {

namespace {

constexpr int kStatMax = 256;  // threads of a row's CTA

// Sum over t < kStatMax of val(t), by one warp, in block_sum's order; in all lanes.
// Each level adds only the pairs that go on: two registers' halves change places
// in the shuffle, so that 4, 2, then 1 register hold them.
template <class Val>
__device__ __forceinline__ double warp_tree(Val val) {
  static_assert(kStatMax == 256, "eight warps' trees");
  const int lane = threadIdx.x & 31;
  double a[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int i = g * 32 + lane, t = (i >> 4) * 32 + (i & 15);
    a[g] = val(t) + val(t + 16);
  }
  auto fold = [lane](double u, double v, int o) {
    return ((lane & o) ? v : u) + __shfl_xor_sync(0xffffffffu, (lane & o) ? u : v, o);
  };
  double c = fold(fold(a[0], a[1], 8), fold(a[2], a[3], 8), 4);
  // within a warp's sum 2 and 1, then between the warps (their index's bits 2, 1, 0
  // are the lane's bits 2, 3, 4)
#pragma unroll
  for (int o : {2, 1, 4, 8, 16}) c += __shfl_xor_sync(0xffffffffu, c, o);
  return c;
}

// Row i of X: its mean, the means of its lag windows and a pass over the centred
// values: each(t, x_t - mean) for every t < n in the thread's order.
// Window s = p - b is [s, s + n - p), its sum taken over threads that each add
// every 256th sample from s + thread on, and then a tree.  (The order is fixed: an
// ulp of a window mean flips the last bits of the normal equations and with them
// FP32 roundings of the fitted lag matrices.)  Those samples are the ones that
// thread + s adds in window 0, and at most one more at the end, so one pass serves
// every window: w, the thread's samples below n - p; w1, the same without the
// first, which stands for thread + s >= 256; the sample at the end apart.  m = 203,
// n = 4001, p = 3: 3 FP64 instructions a sample for 9 with a pass per window, the
// VAR fit 912 us for 930.
template <class Each>
__device__ __forceinline__ void centre_row(const double* __restrict__ x, int m, int n, int p,
                                           double inv_n, double inv_eff, double* red,
                                           double* __restrict__ mu_out,
                                           double* __restrict__ wbar, int* st, Each each) {
  const int i = blockIdx.x, tid = threadIdx.x;
  double s = 0.0;
  bool finite = true;
#pragma unroll 4
  for (int t = tid; t < n; t += kStatMax) {
    const double v = x[t];
    finite &= is_finite(v);
    s += v;
  }
  if (__syncthreads_or(!finite) && tid == 0) set_status(st, VL_ERR_NONFINITE);
  const double mu = block_sum(s, red, [n, inv_n](double t) { return div_by(t, n, inv_n); });
  if (tid == 0) mu_out[i] = mu;
  const int n_eff = n - p;
  __shared__ double w0s[kStatMax], w1s[kStatMax], ends[kStatMax];
  double w = 0.0, w1 = 0.0, end = 0.0;
#pragma unroll 4
  for (int t = tid; t < n; t += kStatMax) {
    const double d = x[t] - mu;
    if (t < n_eff) {
      w += d;
      if (tid < p && t != tid) w1 += d;
    } else {
      end = d;
    }
    each(t, d);
  }
  w0s[tid] = w;
  w1s[tid] = w1;
  ends[tid] = end;
  __syncthreads();
  if (p < kStatMax) {
    for (int sh = tid >> 5; sh <= p; sh += kStatMax / 32) {  // a warp per window
      const double sum = warp_tree([&](int t) {
        const int j = (t + sh) & (kStatMax - 1);
        const int e = j + (n_eff - j + kStatMax - 1) / kStatMax * kStatMax;  // first >= n_eff
        double v = t + sh < kStatMax ? w0s[j] : w1s[j];
        if (e < n_eff + sh) v += ends[j];
        return v;
      });
      if ((tid & 31) == 0) wbar[(int64_t)(p - sh) * m + i] = div_by(sum, n_eff, inv_eff);
    }
    return;
  }
  for (int b = 0; b <= p; ++b) {
    w = 0.0;
    for (int t = tid; t < n_eff; t += kStatMax) w += x[p - b + t] - mu;
    w = block_sum(w, red);
    if (tid == 0) wbar[(int64_t)b * m + i] = div_by(w, n_eff, inv_eff);
  }
}

__global__ void __launch_bounds__(kStatMax)
    var_prep_kernel(const double* __restrict__ X, int64_t ldx, int m, int n, int p, double inv_n,
                    double inv_eff, double* __restrict__ Xc, int64_t ldc,
                    double* __restrict__ mu_out, double* __restrict__ wbar, int* st) {
  pdl_begin(X, Xc, mu_out, wbar, st);
  __shared__ double red[2 * kStatMax];
  double* xc = Xc + blockIdx.x * ldc;
  centre_row(X + blockIdx.x * ldx, m, n, p, inv_n, inv_eff, red, mu_out, wbar, st,
             [xc](int t, double d) { xc[t] = d; });
  for (int t = n + threadIdx.x; t < ldc; t += blockDim.x) xc[t] = 0.0;
}

// Mixed path: the centred series as FP32 (Xc), and the slices of its lag windows:
// row b m + k of W is Xc[k][p - b + t], t < n_eff, for b = 0..p (b = 0 is Y, b =
// tau is Z_tau); S[z][row][k] (row stride ldo, plane stride plane, zeros for
// n_eff <= t < Kpad).  One block per variable k; one exponent per variable for all
// of its windows, and each sample sliced once for all of them.
__global__ void __launch_bounds__(kStatMax)
    prep_lags_kernel(const double* __restrict__ X, int64_t ldx, int m, int n, int p, double inv_n,
                     double inv_eff, float* __restrict__ Xc, int64_t ldc,
                     double* __restrict__ mu_out, double* __restrict__ wbar, int Kpad,
                     __nv_bfloat16* __restrict__ S, int64_t ldo, int64_t plane,
                     int* __restrict__ exps, int* st) {
  pdl_begin(X, Xc, mu_out, wbar, S, exps, st);
  __shared__ double red[2 * kStatMax];
  __shared__ unsigned long long redu[32];
  const int k = blockIdx.x, n_eff = n - p;
  float* xc = Xc + k * ldc;
  uint32_t mx = 0;
  centre_row(X + k * ldx, m, n, p, inv_n, inv_eff, red, mu_out, wbar, st, [&](int t, double d) {
    const float f = bits::to_float(d);
    mx = max(mx, __float_as_uint(f) & 0x7fffffffu);
    xc[t] = f;
  });
  for (int t = n + threadIdx.x; t < ldc; t += blockDim.x) xc[t] = 0.f;
  // float bits: f < 2^(E - 126) for biased exponent E (0 -> 0)
  const unsigned long long fb = block_max_u64(mx, redu);
  const int ex = fb == 0 ? 0 : clamp_exp((int)((fb >> 23) & 0xff) - 126);
  const float sc = ldexpf(1.f, 7 - ex);
  for (int b = threadIdx.x; b <= p; b += blockDim.x) exps[b * m + k] = ex;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {  // the thread's own xc[t]
    __nv_bfloat16 s0, s1, s2;
    slice3(xc[t] * sc, 0.f, s0, s1, s2);
    for (int b = 0; b <= p; ++b) {
      const int u = t - (p - b);
      if (u < 0 || u >= n_eff) continue;
      __nv_bfloat16* o = S + (int64_t)(b * m + k) * ldo + u;
      o[0] = s0;
      o[plane] = s1;
      o[2 * plane] = s2;
    }
  }
  const __nv_bfloat16 z = __float2bfloat16_rn(0.f);
  for (int b = 0; b <= p; ++b)
    for (int t = n_eff + threadIdx.x; t < Kpad; t += blockDim.x) {
      __nv_bfloat16* o = S + (int64_t)(b * m + k) * ldo + t;
      o[0] = z;
      o[plane] = z;
      o[2 * plane] = z;
    }
}

// Centred normal equations of the VAR: G holds, for the Z rows a = (tau-1) m + k
// against every W row b (W = [Y; Z_1; ..; Z_p], windows of the series centred
// by its full mean), the raw cross-product; the intercept is removed by the
// rank-one window-mean correction n_eff * wbar_a * wbar_b.
template <class T>
__global__ void var_normal_eq_kernel(const double* __restrict__ G, int m, int p, int n_eff,
                                     const double* __restrict__ wbar, T* __restrict__ Gzz,
                                     T* __restrict__ Gzy, float* __restrict__ nhi,
                                     float* __restrict__ nlo) {
  pdl_begin(G, wbar, Gzz, Gzy, nhi, nlo);
  const int mp = m * p, q = m * (p + 1);
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)mp * q) return;
  const int a = (int)(idx / q), b = (int)(idx % q);
  const double v = G[idx] - (double)n_eff * wbar[m + a] * wbar[b];
  if (nhi) {  // the same values as an FP32 pair, for the refinement residual
    const float h = (float)v;
    nhi[idx] = h;
    nlo[idx] = (float)(v - (double)h);
  }
  if (b < m)
    Gzy[(int64_t)a * m + b] = (T)v;
  else
    Gzz[(int64_t)a * mp + (b - m)] = (T)v;
}

template <class T>
__global__ void var_coef_kernel(const T* __restrict__ beta, int m, int p, double* __restrict__ M) {
  pdl_begin(beta, M);
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)p * m * m) return;
  const int tau = (int)(idx / ((int64_t)m * m));
  const int rem = (int)(idx % ((int64_t)m * m));
  const int i = rem / m, k = rem % m;
  M[idx] = (double)beta[((int64_t)tau * m + k) * m + i];
}

// cst[i] = wbar0_i - sum_a beta[a][i] wbar_{Z,a}: a CTA takes CST_C columns i, the
// rows a dealt to the rest of its threads (consecutive threads on consecutive
// columns; one warp per column read beta with a stride of m).
constexpr int CST_C = 16, CST_TH = 512;
template <class T>
__global__ void __launch_bounds__(CST_TH)
    var_cst_kernel(const T* __restrict__ beta, int m, int p, const double* __restrict__ wbar,
                   double* __restrict__ cst) {
  pdl_begin(beta, wbar, cst);
  __shared__ double red[CST_TH / 32][CST_C];
  const int i = blockIdx.x * CST_C + threadIdx.x % CST_C;
  double c = 0.0;
  if (i < m)
    for (int a = threadIdx.x / CST_C; a < m * p; a += CST_TH / CST_C) {
      const T v = beta[(int64_t)a * m + i];
      if constexpr (sizeof(T) == 4)
        c = fma(bits::to_double(v), wbar[m + a], c);
      else
        c = fma(v, wbar[m + a], c);
    }
  c += __shfl_xor_sync(0xffffffffu, c, CST_C);
  if ((threadIdx.x & 31) < CST_C) red[threadIdx.x >> 5][threadIdx.x % CST_C] = c;
  __syncthreads();
  if (threadIdx.x < CST_C && i < m) {
    double t = 0.0;
    for (int w = 0; w < CST_TH / 32; ++w) t += red[w][threadIdx.x];
    cst[i] = wbar[i] - t;
  }
}

__global__ void var_resid_init_kernel(const double* __restrict__ X, int64_t ldx, int n_eff, int p,
                                      const double* __restrict__ mu,
                                      const double* __restrict__ cst, double* __restrict__ E,
                                      int64_t lde) {
  pdl_begin(X, mu, cst, E);
  const int i = blockIdx.y;
  const double off = mu[i] + cst[i];
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_eff; t += gridDim.x * blockDim.x)
    E[(int64_t)i * lde + t] = X[(int64_t)i * ldx + p + t] - off;
}

__device__ __forceinline__ void kahan_f(float& S, float& C, float x) {
  float y = x - C;
  float t = S + y;
  C = (t - S) - y;
  S = t;
}

// Mean, then 1/std (0 for a constant row) of row e; each(d) sees every centred
// value between the two.  Sets the status word for rows that are not finite or
// constant and goes on (a row that is not finite leaves NaN everywhere).  The mean
// is the sum in block_sum's order, divided: n copies of a number with an exact sum
// have that number as their mean, and a variance of exactly 0.
template <class Each>
__device__ __forceinline__ void row_stats(const double* __restrict__ e, int n, double inv_n,
                                          double* red, int* st, double& mu, double& isd,
                                          Each each) {
  double s = 0.0;
  bool finite = true;
#pragma unroll 4
  for (int t = threadIdx.x; t < n; t += kStatMax) {
    const double v = e[t];
    finite &= is_finite(v);
    s += v;
  }
  if (__syncthreads_or(!finite) && threadIdx.x == 0) set_status(st, VL_ERR_NONFINITE);
  mu = block_sum(s, red, [n, inv_n](double t) { return div_by(t, n, inv_n); });
  double q = 0.0;
#pragma unroll 4
  for (int t = threadIdx.x; t < n; t += kStatMax) {
    const double d = e[t] - mu;
    q += d * d;
    each(d);
  }
  isd = block_fold(q, red, [inv_n, st](double t) {
    const double var = t * inv_n;
    if (var > 1e-300 || var != var) return rsqrt(var);
    set_status(st, VL_ERR_DEGENERATE);
    return 0.0;
  });
}

// H of a standardized row from the block's sums of log cosh u and u e^{-u^2/2};
// a constant row counts as moments 0.
__device__ __forceinline__ void store_entropy(double a, double b, double inv_n, double isd,
                                              double* red, double* __restrict__ hx) {
  block_sum2(a, b, red);
  if (threadIdx.x == 0)
    *hx = isd == 0.0 ? entropy_from_moments(0.0, 0.0)
                     : entropy_from_moments(a * inv_n, b * inv_n);
}

__global__ void __launch_bounds__(kStatMax)
    standardize_kernel(const double* __restrict__ E, int64_t lde, int n, double inv_n,
                       double* __restrict__ mu_out, double* __restrict__ isd_out,
                       double* __restrict__ hx, int* st) {
  pdl_begin(E, mu_out, isd_out, hx, st);
  __shared__ double red[2 * kStatMax];
  __shared__ fx::u64 te[fx::EXP_N], tl[fx::LOG_N];
  __shared__ fx::u32 tr[fx::LOG_N];
  const fx::Tab tab{te, tl, tr};
  if (hx) fx::fill_tables(te, tl, tr);
  const int i = blockIdx.x;
  const double* e = E + (int64_t)i * lde;
  double mu, isd;
  row_stats(e, n, inv_n, red, st, mu, isd, [](double) {});
  if (threadIdx.x == 0) {
    mu_out[i] = mu;
    isd_out[i] = isd;
  }
  if (!hx) return;
  // fixed-point functions and exact sums (fx64.cuh) of kappa times the value the
  // pairwise kernel reads, so that H(x_i) and the residuals' entropies share the
  // rounding of 1/std, which D's differences then cancel
  fx::Moments M;
  int cnt = 0;
  double a, b;
  for (int t = threadIdx.x; t < n; t += blockDim.x, ++cnt)
    fx::moments_add(M, fx::KAPPA64 * ((e[t] - mu) * isd), tab);
  fx::moments_sums(M, cnt, a, b);
  store_entropy(a, b, inv_n, isd, red, hx + i);
}

// Mixed path, one block per row: statistics and entropy, the slices of the
// centred row (S[z][i][k], k < K; zeros up to Kpad) with its exponent, and the
// standardized row as FP32, to xs[i][t] (row stride n_pad) or, time-major, to
// xt[t][i] (row stride m_pad; the blocks i >= m write its zero columns).  FULL =
// false: the slices only (and the checks of the statistics).
template <bool FULL>
__global__ void __launch_bounds__(kStatMax)
    measure_prep_kernel(const double* __restrict__ E, int64_t lde, int m, int n, double inv_n,
                        int Kpad,
                        __nv_bfloat16* __restrict__ S, int64_t plane, int* __restrict__ exps,
                        float* __restrict__ xs, float* __restrict__ xt, int m_pad, int n_pad,
                        double* __restrict__ hx, int* st) {
  pdl_begin(E, S, exps, xs, xt, hx, st);
  __shared__ double red[2 * kStatMax];
  __shared__ unsigned long long redu[32];
  const int i = blockIdx.x;
  if (i >= m) {
    for (int t = threadIdx.x; t < n_pad; t += blockDim.x) xt[(int64_t)t * m_pad + i] = 0.f;
    return;
  }
  const double* e = E + (int64_t)i * lde;
  double mu, isd;
  unsigned long long mx = 0;
  row_stats(e, n, inv_n, red, st, mu, isd, [&mx](double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d) & 0x7fffffffffffffffull;
    mx = b > mx ? b : mx;
  });
  const int ex = exp_above(block_max_u64(mx, redu));
  if (threadIdx.x == 0) exps[i] = ex;
  const float sc = ldexpf(1.f, 7 - ex);
  __nv_bfloat16* o = S + (int64_t)i * Kpad;
  // FP32 per-sample functions (CUDA's accurate expf / log1pf), Kahan sums of log
  // cosh u + ln 2 (= |u| + log1p(e^{-2|u|})) and u e^{-u^2/2}
  float sa = 0.f, ca = 0.f, sb = 0.f, cb = 0.f;
  int cnt = 0;
  for (int t = threadIdx.x; t < n; t += blockDim.x, ++cnt) {
    const double d = e[t] - mu;
    const float h = bits::to_float(d);
    const float l = bits::to_float(d - bits::to_double(h));
    __nv_bfloat16 s0, s1, s2;
    slice3(h * sc, l * sc, s0, s1, s2);
    o[t] = s0;
    o[plane + t] = s1;
    o[2 * plane + t] = s2;
    if constexpr (!FULL) continue;
    const float u = bits::to_float(d * isd);
    if (xs)
      xs[(int64_t)i * n_pad + t] = u;
    else
      xt[(int64_t)t * m_pad + i] = u;
    const float au = fabsf(u);
    kahan_f(sa, ca, au + log1pf(expf(-2.0f * au)));
    kahan_f(sb, cb, u * expf(-0.5f * u * u));
  }
  const __nv_bfloat16 z = __float2bfloat16_rn(0.f);
  for (int t = n + threadIdx.x; t < Kpad; t += blockDim.x) o[t] = o[plane + t] = o[2 * plane + t] = z;
  if constexpr (!FULL) return;
  for (int t = n + threadIdx.x; t < n_pad; t += blockDim.x) {
    if (xs)
      xs[(int64_t)i * n_pad + t] = 0.f;
    else
      xt[(int64_t)t * m_pad + i] = 0.f;
  }
  store_entropy((bits::to_double(sa) - bits::to_double(ca)) - LN2 * cnt,
                bits::to_double(sb) - bits::to_double(cb), inv_n, isd, red, hx + i);
}

__global__ void center64_kernel(const double* __restrict__ E, int64_t lde, int n,
                                const double* __restrict__ mu, double* __restrict__ out,
                                int64_t ldc) {
  pdl_begin(E, mu, out);
  const int i = blockIdx.y;
  const double mi = mu[i];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ldc;
       t += (int64_t)gridDim.x * blockDim.x)
    out[(int64_t)i * ldc + t] = (t < n) ? E[(int64_t)i * lde + t] - mi : 0.0;
}

// 32 x 32 tiled transpose: xt[t * m_pad + i] = (E[i, t] - mu_i) / sd_i.
__global__ void transpose_std_kernel(const double* __restrict__ E, int64_t lde, int m, int n,
                                     const double* __restrict__ mu,
                                     const double* __restrict__ isd, double* __restrict__ xt,
                                     int m_pad, int n_pad) {
  pdl_begin(E, mu, isd, xt);
  __shared__ double tile[32][33];
  const int t0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int r = ty; r < 32; r += 8) {
    int i = i0 + r, t = t0 + tx;
    tile[r][tx] = (i < m && t < n) ? (E[(int64_t)i * lde + t] - mu[i]) * isd[i] : 0.0;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    int t = t0 + r, i = i0 + tx;
    if (t < n_pad && i < m_pad) xt[(int64_t)t * m_pad + i] = tile[tx][r];
  }
}

// xt[t * m_pad + i] = xs[i * n_pad + t] (zero for i >= m); n_pad and m_pad are
// multiples of 32.
__global__ void transpose_f32_kernel(const float* __restrict__ xs, int m, int n_pad,
                                     float* __restrict__ xt, int m_pad) {
  pdl_begin(xs, xt);
  __shared__ float tile[32][33];
  const int t0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
#pragma unroll
  for (int r = ty; r < 32; r += 8)
    tile[r][tx] = i0 + r < m ? xs[(int64_t)(i0 + r) * n_pad + t0 + tx] : 0.f;
  __syncthreads();
#pragma unroll
  for (int r = ty; r < 32; r += 8) xt[(int64_t)(t0 + r) * m_pad + i0 + tx] = tile[tx][r];
}

}  // namespace

void launch_var_prep(const double* X, int64_t ldx, int m, int n, int p, double* Xc, int64_t ldc,
                     double* mu, double* wbar, int* st, Lane s) {
  launch(var_prep_kernel, m, kStatMax, 0, s, X, ldx, m, n, p, 1.0 / n,
         1.0 / (n - p), Xc, ldc, mu, wbar, st);
}

void launch_prep_lags(const double* X, int64_t ldx, int m, int n, int p, float* Xc, int64_t ldc,
                      double* mu, double* wbar, int64_t Kpad, void* S, int64_t plane, int* exps,
                      int* st, Lane s) {
  launch(prep_lags_kernel, m, kStatMax, 0, s, X, ldx, m, n, p, 1.0 / n,
         1.0 / (n - p), Xc, ldc, mu, wbar,
         (int)Kpad, static_cast<__nv_bfloat16*>(S), Kpad, plane, exps, st);
}

template <class T>
void launch_var_normal_eq(const double* G, int m, int p, int n_eff, const double* wbar, T* Gzz,
                          T* Gzy, Lane s, float* nhi, float* nlo) {
  const int mp = m * p;
  const int64_t tot = (int64_t)mp * (mp + m);
  launch(var_normal_eq_kernel<T>, (unsigned)((tot + 255) / 256), 256, 0, s, G, m, p, n_eff, wbar,
         Gzz, Gzy, nhi, nlo);
}
template void launch_var_normal_eq<float>(const double*, int, int, int, const double*, float*,
                                          float*, Lane, float*, float*);
template void launch_var_normal_eq<double>(const double*, int, int, int, const double*,
                                           double*, double*, Lane, float*, float*);

template <class T>
void launch_var_coef(const T* beta, int m, int p, const double* wbar, double* M, double* cst,
                     Lane s) {
  const int64_t tot = (int64_t)p * m * m;
  launch(var_coef_kernel<T>, (unsigned)((tot + 255) / 256), 256, 0, s, beta, m, p, M);
  launch(var_cst_kernel<T>, (m + CST_C - 1) / CST_C, CST_TH, 0, s, beta, m, p, wbar, cst);
}
template void launch_var_coef<float>(const float*, int, int, const double*, double*, double*,
                                     Lane);

template <class T>
void launch_var_cst(const T* beta, int m, int p, const double* wbar, double* cst, Lane s) {
  launch(var_cst_kernel<T>, (m + CST_C - 1) / CST_C, CST_TH, 0, s, beta, m, p, wbar, cst);
}
template void launch_var_cst<float>(const float*, int, int, const double*, double*, Lane);
template void launch_var_coef<double>(const double*, int, int, const double*, double*, double*,
                                      Lane);

void launch_var_resid_init(const double* X, int64_t ldx, int m, int n, int p, const double* mu,
                           const double* cst, double* E, int64_t lde, Lane s) {
  const int n_eff = n - p;
  dim3 grid((unsigned)((n_eff + 255) / 256 < 64 ? (n_eff + 255) / 256 : 64), m);
  launch(var_resid_init_kernel, grid, 256, 0, s, X, ldx, n_eff, p, mu, cst, E, lde);
}

void launch_standardize(const double* E, int64_t lde, int m, int n, double* mu, double* inv_sd,
                        double* hx, int* st, Lane s) {
  launch(standardize_kernel, m, kStatMax, 0, s, E, lde, n, 1.0 / n, mu, inv_sd, hx, st);
}

// The standardized rows go straight to their time-major places while that is
// little traffic (each four bytes then write a 32-byte sector), through xs and a
// transpose beyond: at m n = 2^19 both take about 5 us.
constexpr int64_t kDirectMax = 1 << 19;

bool measure_prep_needs_rows(int m, int n) { return (int64_t)m * n > kDirectMax; }

void launch_measure_prep(const double* E, int64_t lde, int m, int n, int64_t Kpad, void* S,
                         int64_t plane, int* exps, float* xs, float* xt, int m_pad, int n_pad,
                         double* hx, int* st, Lane s) {
  __nv_bfloat16* Sb = static_cast<__nv_bfloat16*>(S);
  if (!xt) {
    launch(measure_prep_kernel<false>, m, kStatMax, 0, s, E, lde, m, n, 1.0 / n, (int)Kpad, Sb,
           plane, exps, nullptr, nullptr, 0, 0, nullptr, st);
    return;
  }
  const bool rows = measure_prep_needs_rows(m, n);
  launch(measure_prep_kernel<true>, rows ? m : m_pad, kStatMax, 0, s, E, lde, m, n, 1.0 / n,
         (int)Kpad, Sb, plane, exps, rows ? xs : nullptr, xt, m_pad, n_pad, hx, st);
  if (rows) {
    launch(transpose_f32_kernel, dim3(n_pad / 32, m_pad / 32), dim3(32, 8), 0, s, xs, m, n_pad, xt,
           m_pad);
  }
}

void launch_center64(const double* E, int64_t lde, int m, int n, const double* mu, double* out,
                     int64_t ldc, Lane s) {
  dim3 grid((unsigned)((ldc + 255) / 256 < 64 ? (ldc + 255) / 256 : 64), m);
  launch(center64_kernel, grid, 256, 0, s, E, lde, n, mu, out, ldc);
}

void launch_transpose_std(const double* E, int64_t lde, int m, int n, const double* mu,
                          const double* inv_sd, double* xt, int m_pad, int n_pad,
                          Lane s) {
  dim3 grid((n_pad + 31) / 32, (m_pad + 31) / 32), block(32, 8);
  launch(transpose_std_kernel, grid, block, 0, s, E, lde, m, n, mu, inv_sd, xt, m_pad, n_pad);
}

namespace {

// One CTA: 2 sum ln L[i][i] in FP64 (a fixed-order block reduction).
__global__ void logdet_value_kernel(const double* __restrict__ L, int64_t ldl, int m,
                                    double penalty, double* __restrict__ value, int* st) {
  pdl_begin(L, value, st);
  __shared__ double red[2 * kStatMax];
  double s = 0.0;
  bool bad = false;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const double d = L[(int64_t)i * ldl + i];
    bad |= !(d > 0.0);
    s += d > 0.0 ? log(d) : 0.0;
  }
  if (__syncthreads_or(bad)) {
    if (threadIdx.x == 0) set_status(st, VL_ERR_RANK);
    return;
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) *value = 2.0 * s + penalty;
}

__global__ void argmin_p_kernel(const double* __restrict__ values, int p_max,
                                int32_t* __restrict__ p_best) {
  pdl_begin(values, p_best);
  int best = 0;
  for (int i = 1; i < p_max; ++i)
    if (values[i] < values[best]) best = i;
  *p_best = best + 1;
}

}  // namespace

void launch_logdet_value(const double* L, int64_t ldl, int m, double penalty, double* value,
                         int* st, Lane s) {
  launch(logdet_value_kernel, 1, kStatMax, 0, s, L, ldl, m, penalty, value, st);
}

void launch_argmin_p(const double* values, int p_max, int32_t* p_best, Lane s) {
  launch(argmin_p_kernel, 1, 1, 0, s, values, p_max, p_best);
}

}  // namespace vl
