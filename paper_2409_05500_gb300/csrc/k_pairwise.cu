// The one-time O(m^2 n) pairwise precomputation (Sec. 4.2 items 1-2 and
// Algorithm 1's two precompute calls; Eqs. 1-2 of Sec. 3).
//
// For every unordered pair i < j and every sample t the two standardized
// regression residuals are
//     u_t = s (x_i[t] - rho x_j[t]),   v_t = s (x_j[t] - rho x_i[t]),
//     s = (1 - rho^2)^{-1/2},
// and H needs, per residual, A = mean log cosh u and B = mean u exp(-u^2/2).
//
// FP32 kernel arithmetic (per residual stream, per sample):
//     w    = kappa s r                  kappa = 2 log2(e), so 2^{-|w|} = e^{-2|u|}
//     y    = ex2(-|w|)                  (MUFU)
//     prod = prod * (1 + y)             log cosh u = |u| + ln(1 + y) - ln 2
//     ra  += |w|
//     g    = ex2(-w^2 / (8 log2 e))     = e^{-u^2/2}   (MUFU)
//     rb  += w g
// Every KRUN = 16 samples the run's log-cosh sum
//     sum_t log cosh u_t = ra / kappa + ln 2 (log2(prod) - 16)
// (one MUFU lg2 per run) and its sb are Kahan-added into FP32 (sum, comp)
// pairs.  The two j's of a thread's micro-tile are processed as one float2
// with the paired FP32 instructions of this architecture (fma/mul/add .f32x2),
// which halves the FP32 instruction count; the exponentials stay scalar MUFU.
// The split partials are combined in double-float arithmetic by
// measure_finalize.
//
// Padding: x is zero beyond n (time) and beyond m (variables).  A zero sample
// gives |w| = 0, 1 + y = 2 (log2 adds exactly 1, cancelled by the -16 per
// run) and w g = 0, i.e. it contributes exactly 0: padding needs no masking.
#include <algorithm>
#include <cmath>

#include "fp64_bits.cuh"
#include "fx64.cuh"
#include "vl_internal.cuh"

namespace vl {

namespace {

constexpr int TB = 32;        // variables per tile side
constexpr int KRUN = 16;      // samples per product/Kahan run (product <= 2^16)
constexpr float KAPPA = 2.8853900817779268f;       // 2 log2(e)
constexpr float GAUSS_K = -0.08664339756999316f;   // -1 / (8 log2 e)

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// tile index -> (I, J), I <= J, row-major over the upper triangle
__device__ __forceinline__ void tile_coords(int q, int T, int& I, int& J) {
  // row i starts at i (2 T - i + 1) / 2
  const float w = 2.f * T + 1.f;
  int i = max(0, min((int)((w - sqrtf(fmaxf(w * w - 8.f * (float)q, 0.f))) * 0.5f), T - 1));
  while (i > 0 && i * (2 * T - i + 1) / 2 > q) --i;
  while ((i + 1) * (2 * T - i) / 2 <= q) ++i;
  I = i;
  J = i + q - i * (2 * T - i + 1) / 2;
}

// State of two residual streams (the two j's of a micro-tile row), as float2.
struct Pair2 {
  float2 prod, ra, rb;      // current 16-sample run
  float2 sa, ca, sb, cb;    // Kahan (sum, compensation) of the run sums
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// (S, C) += x, Kahan, both lanes at once
__device__ __forceinline__ void kahan2(float2& S, float2& C, float2 x) {
  const float2 mone = f2(-1.f, -1.f);
  const float2 y = __ffma2_rn(C, mone, x);  // x - C
  const float2 t = __fadd2_rn(S, y);
  C = __ffma2_rn(y, mone, __ffma2_rn(S, mone, t));  // (t - S) - y
  S = t;
}

// Thread -> MTI x 2 pair micro-tile (ti, tj) of tile (I, J), enumerating only
// micro-tiles holding at least one pair i < j < m; returns false for threads
// beyond that count.  Micro-tile (ti, tj) covers i = MTI ti + a, j = 2 tj + b.
template <int MTI>
__device__ __forceinline__ bool micro_tile(int s, int I, int J, int m, int& ti, int& tj) {
  constexpr int R = TB / MTI;                     // micro-rows
  const int lim = min(16, (m - J * TB + 1) / 2);  // micro-columns with some j < m
  if (I < J) {
    ti = s / lim;
    tj = s % lim;
    if (ti < R) return true;
  } else {
    // diagonal tile: row ti needs 2 tj + 1 > MTI ti, i.e. tj >= (MTI ti + 1) / 2
    for (int r = 0; r < R; ++r) {
      const int st = (MTI * r + 1) / 2;
      const int len = lim - st;
      if (len <= 0) break;
      if (s < len) {
        ti = r;
        tj = st + s;
        return true;
      }
      s -= len;
    }
  }
  ti = 0;
  tj = 0;
  return false;
}

// One sample of one stream pair: residual R (both lanes), scale C.
__device__ __forceinline__ void step2(Pair2& q, float2 R, float2 C, float2 KK) {
  const float2 W = __fmul2_rn(C, R);
  const float2 Y = f2(ex2_approx(-fabsf(W.x)), ex2_approx(-fabsf(W.y)));
  q.prod = __ffma2_rn(q.prod, Y, q.prod);
  q.ra.x += fabsf(W.x);
  q.ra.y += fabsf(W.y);
  const float2 E = __fmul2_rn(__fmul2_rn(W, KK), W);
  const float2 G = f2(ex2_approx(E.x), ex2_approx(E.y));
  q.rb = __ffma2_rn(W, G, q.rb);
}

__device__ __forceinline__ void end_run2(Pair2& q) {
  const float2 L = f2(lg2_approx(q.prod.x), lg2_approx(q.prod.y));
  const float ik = 1.f / KAPPA;
  const float m16 = -16.f * 0.69314718055994531f;
  // sum log cosh over the run = ra / kappa + ln 2 (log2 prod - 16)
  const float2 run =
      __ffma2_rn(L, f2(0.69314718055994531f, 0.69314718055994531f),
                 __ffma2_rn(q.ra, f2(ik, ik), f2(m16, m16)));
  kahan2(q.sa, q.ca, run);
  kahan2(q.sb, q.cb, q.rb);
  q.prod = f2(1.f, 1.f);
  q.ra = f2(0.f, 0.f);
  q.rb = f2(0.f, 0.f);
}

// MTI x 2 pair micro-tiles, (32 / MTI) x 16 threads per 32 x 32 tile, TTS
// samples per shared-memory stage, MINB CTAs per SM.
// One work item: pair tile `tile` of the upper triangle, sample split `split`.
template <int MTI, int TTS>
__device__ __forceinline__ void pairwise_f32_item(int tile, int split,
                                                  const float* __restrict__ xt, int m, int m_pad,
                                                  int T, int n_run, int tps,
                                                  const float* __restrict__ rho32,
                                                  const float* __restrict__ c32,
                                                  float* __restrict__ part) {
  constexpr int NT = TB / MTI * 16;
  extern __shared__ __align__(16) float pw_smem[];
  float(*sx)[TTS][2 * TB] = reinterpret_cast<float(*)[TTS][2 * TB]>(pw_smem);  // [3][TTS][64]
  int I, J;
  tile_coords(tile, T, I, J);
  const int t0 = split * tps;
  const int t1 = min(n_run, t0 + tps);

  // Valid micro-tiles first: on a diagonal tile only those with some i < j,
  // on the last tile column only j < m; threads past the valid count (whole
  // warps, at the end) skip the arithmetic and only help stage the samples.
  int ti, tj;
  const bool active = micro_tile<MTI>(threadIdx.x, I, J, m, ti, tj);
  const int li = MTI * ti, lj = 2 * tj;
  const int gi0 = I * TB + li, gj0 = J * TB + lj;

  // pair (a, b) = (i0 + a, j0 + b); constants as float2 over b
  float2 NR[MTI], C[MTI];
  bool valid[MTI][2];
#pragma unroll
  for (int a = 0; a < MTI; ++a) {
    float r2[2], c2[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int gi = gi0 + a, gj = gj0 + b;
      valid[a][b] = active && (gi < gj) && (gj < m);
      r2[b] = valid[a][b] ? rho32[(int64_t)gi * m + gj] : 0.f;
      c2[b] = valid[a][b] ? c32[(int64_t)gi * m + gj] : KAPPA;
    }
    NR[a] = f2(-r2[0], -r2[1]);
    C[a] = f2(c2[0], c2[1]);
  }
  const float2 KK = f2(GAUSS_K, GAUSS_K);
  // stream pairs: 2a = residuals of i_a on (j0, j1), 2a + 1 = of (j0, j1) on i_a
  Pair2 q[2 * MTI];
#pragma unroll
  for (int k = 0; k < 2 * MTI; ++k)
    q[k] = Pair2{f2(1.f, 1.f), f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f),
                 f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f)};

  // stage loader: TTS rows x (32 + 32) floats = TTS * 16 chunks of 16 B
  auto load_stage = [&](int buf, int tb) {
    for (int idx = threadIdx.x; idx < TTS * 16; idx += NT) {
      const int r = idx >> 4, c = idx & 15;  // c: 0-7 I block, 8-15 J block
      const int t = tb + r;
      if (t < t1) {
        const int col = (c < 8) ? (I * TB + 4 * c) : (J * TB + 4 * (c - 8));
        cp_async16(&sx[buf][r][4 * c], xt + (int64_t)t * m_pad + col);
      }
    }
    cp_async_commit();
  };

  // three-stage ring: stage s+2 is copied while stage s is consumed, and the
  // one barrier per stage both publishes stage s and frees the buffer of
  // stage s-1 for the copy of stage s+2
  const int nst = t1 > t0 ? (t1 - t0 + TTS - 1) / TTS : 0;
  if (nst > 0) load_stage(0, t0);
  if (nst > 1) load_stage(1, t0 + TTS);
  for (int st = 0; st < nst; ++st) {
    const int tb = t0 + st * TTS, buf = st % 3;
    const int rows = min(TTS, t1 - tb);
    if (st + 1 < nst)
      cp_async_wait<1>();
    else
      cp_async_wait<0>();
    __syncthreads();
    if (st + 2 < nst) load_stage((st + 2) % 3, tb + 2 * TTS);
    for (int r0 = 0; active && r0 < rows; r0 += KRUN) {
#pragma unroll
      for (int k = 0; k < KRUN; ++k) {
        const float2 xj = *reinterpret_cast<const float2*>(&sx[buf][r0 + k][TB + lj]);
        float xi[MTI];
        if constexpr (MTI == 2) {
          const float2 v = *reinterpret_cast<const float2*>(&sx[buf][r0 + k][li]);
          xi[0] = v.x;
          xi[1] = v.y;
        } else {
          xi[0] = sx[buf][r0 + k][li];
        }
#pragma unroll
        for (int a = 0; a < MTI; ++a) {
          const float2 xa = f2(xi[a], xi[a]);
          step2(q[2 * a], __ffma2_rn(NR[a], xj, xa), C[a], KK);      // x_i - rho x_j
          step2(q[2 * a + 1], __ffma2_rn(NR[a], xa, xj), C[a], KK);  // x_j - rho x_i
        }
      }
#pragma unroll
      for (int k = 0; k < 2 * MTI; ++k) end_run2(q[k]);
    }
  }

  // partials of this split as exact double-float pairs (sum, -comp):
  // part[(split*4 + k) * m*m + a*m + b] for the residual of a on b, k = 0, 1:
  // sum of log cosh u; k = 2, 3: sum of w e^{-u^2/2}.  No FP64 arithmetic here.
  const int64_t mm = (int64_t)m * m;
#pragma unroll
  for (int a = 0; a < MTI; ++a) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (!valid[a][b]) continue;
      const int gi = gi0 + a, gj = gj0 + b;
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const Pair2& st = q[2 * a + d];
        const int64_t off = d ? ((int64_t)gj * m + gi) : ((int64_t)gi * m + gj);
        float* base = part + (int64_t)split * 4 * mm + off;
        base[0] = b ? st.sa.y : st.sa.x;
        base[mm] = -(b ? st.ca.y : st.ca.x);
        base[2 * mm] = b ? st.sb.y : st.sb.x;
        base[3 * mm] = -(b ? st.cb.y : st.cb.x);
      }
    }
  }
}

template <int MTI, int TTS, int MINB>
__global__ void __launch_bounds__(TB / MTI * 16, MINB)
    pairwise_f32_kernel(const float* __restrict__ xt, int m, int m_pad, int T, int n_run,
                        int tps, const float* __restrict__ rho32,
                        const float* __restrict__ c32, float* __restrict__ part) {
  // (releasing the finalisation early, whose CTAs then wait beside this one: m = 50,
  // n = 5000 the measure 112 us, 65 as here; m = 100, n = 2600 80 and 59)
  pdl_wait(xt, rho32, c32, part);
  pairwise_f32_item<MTI, TTS>(blockIdx.x, blockIdx.y, xt, m, m_pad, T, n_run, tps, rho32, c32,
                              part);
}

// Many instances in one launch: a device list of (job, tile, split) items,
// ordered by cost (largest first), dealt round-robin to a grid of about one
// CTA per SM; each CTA runs its items one after another.
template <int MTI, int TTS, int MINB>
__global__ void __launch_bounds__(TB / MTI * 16, MINB)
    pairwise_f32_list_kernel(const PairJob* __restrict__ jobs, const int4* __restrict__ items,
                             int nitems) {
  pdl_begin(jobs, items);
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int4 w = items[it];
    const PairJob& j = jobs[w.x];
    pairwise_f32_item<MTI, TTS>(w.y, w.z, j.xt, j.m, j.m_pad, j.T, j.n_run, j.tps, j.rho32,
                                j.c32, j.part);
    __syncthreads();  // the sample stages are reused by the next item
  }
}

// FP64 measure.  The residuals are formed in FP64 (one FMA and one product
// each), the per-sample functions and their sums in 63-bit fixed point
// (fx64.cuh), which is closer to exact than FP64 functions and sums are.
// Bound by instructions: 257 a residual sample, the pipe of the integer products
// 73 % busy, the FP64 pipe (two operations, 40 SM clocks a warp) 64 %.  m = 120,
// n = 9997: 1.50 ms; with CUDA's FP64 exp and log1p, which keep the FP64 pipe
// busy 20 times as long, 33.1 ms.
// One pair a < b per thread, consecutive threads consecutive b (coalesced
// loads of the time-major samples, a broadcast of x_a, no padded tiles), the
// samples split over blockIdx.y.  Partials: k = 0 sum log cosh u, k = 1 sum
// u e^{-u^2/2}.
constexpr int FX_TH = 128;

__device__ __forceinline__ void pair_of(int q, int m, int& a, int& b) {
  // row a of the strict upper triangle starts at a (2 m - a - 1) / 2
  const float w = 2.f * m - 1.f;
  a = (int)((w - sqrtf(fmaxf(w * w - 8.f * (float)q, 0.f))) * 0.5f);
  a = max(0, min(a, m - 2));
  while (a > 0 && (int)((int64_t)a * (2 * m - a - 1) / 2) > q) --a;
  while ((int)((int64_t)(a + 1) * (2 * m - a - 2) / 2) <= q) ++a;
  b = a + 1 + q - (int)((int64_t)a * (2 * m - a - 1) / 2);
}

__global__ void __launch_bounds__(FX_TH)
    pairwise_f64_kernel(const double* __restrict__ xt, int m, int m_pad, int n_real, int tps,
                        const double* __restrict__ rho64, const double* __restrict__ c64,
                        double* __restrict__ part) {
  pdl_begin(xt, rho64, c64, part);
  __shared__ fx::u64 te[fx::EXP_N], tl[fx::LOG_N];
  __shared__ fx::u32 tr[fx::LOG_N];
  const fx::Tab T{te, tl, tr};
  fx::fill_tables(te, tl, tr);
  __syncthreads();
  const int q = blockIdx.x * FX_TH + threadIdx.x;
  if (q >= m * (m - 1) / 2) return;
  int a, b;
  pair_of(q, m, a, b);
  const int split = blockIdx.y;
  const int t0 = split * tps, t1 = min(n_real, t0 + tps);
  const double rho = rho64[(int64_t)a * m + b], c = c64[(int64_t)a * m + b];
  fx::Moments ma, mb;  // residual of a on b, of b on a
  const double* row = xt + (int64_t)t0 * m_pad;
  double xa = t0 < t1 ? row[a] : 0.0, xb = t0 < t1 ? row[b] : 0.0;
  for (int t = t0; t < t1; ++t) {
    const double va = xa, vb = xb;
    row += m_pad;
    if (t + 1 < t1) {
      xa = row[a];
      xb = row[b];
    }
    fx::moments_add(ma, c * (va - rho * vb), T);
    fx::moments_add(mb, c * (vb - rho * va), T);
  }
  const int64_t mm = (int64_t)m * m;
  double* base = part + (int64_t)split * 2 * mm;
  const int64_t ab = (int64_t)a * m + b, ba = (int64_t)b * m + a;
  fx::moments_sums(ma, max(0, t1 - t0), base[ab], base[mm + ab]);
  fx::moments_sums(mb, max(0, t1 - t0), base[ba], base[mm + ba]);
}

// FP64 path: rho_ij = C_ij / sqrt(C_ii C_jj) from the centred cross-product matrix
// C and kappa / sqrt(1 - rho^2), i < j.
__global__ void pair_consts64_kernel(const double* __restrict__ C, int m,
                                     double* __restrict__ rho64, double* __restrict__ c64,
                                     int* st) {
  pdl_begin(C, rho64, c64, st);
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int a = (int)(idx / m), b = (int)(idx % m);
  if (idx >= (int64_t)m * m || b <= a) return;
  double r = C[idx] / sqrt(C[(int64_t)a * m + a] * C[(int64_t)b * m + b]);
  if (!(1.0 - r * r >= DEGENERATE_1MR2)) {
    set_status(st, VL_ERR_DEGENERATE);
    r = 0.0;
  }
  rho64[idx] = r;
  c64[idx] = fx::KAPPA64 / sqrt(1.0 - r * r);
}

// Mixed path: the same constants rounded to FP32.  In FP64 the two roots and two
// divisions of a pair are ~90 instructions at 1.6 per clock per SM.  Instead rho =
// C_ij w_i w_j (w_i = 1 / sqrt(C_ii) comes with C) in two products, accurate to a
// few FP64 ulp, and kappa / sqrt(1 - rho^2) in double-float FP32 arithmetic to
// 2^-40; where either lies too close to the middle of two FP32 numbers for its
// rounding to be certain (about one pair in 2,000), or 1 - rho^2 is below 2^-8, the
// pair takes the FP64 expressions.  So every constant is the rounding of the FP64
// expression.  m = 1600: 24 us against 177.
__global__ void pair_consts_kernel(const double* __restrict__ C, const double* __restrict__ w,
                                   int m, float* __restrict__ rho32, float* __restrict__ c32,
                                   int* st) {
  pdl_begin(C, w, rho32, c32, st);
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int a = (int)(idx / m), b = (int)(idx % m);
  if (idx >= (int64_t)m * m || b <= a) return;  // the pairwise kernel reads i < j
  const double cab = C[idx];
  const double ra = cab * (w[a] * w[b]);
  const float hi = bits::to_float(ra);
  const float lo = bits::to_float(ra - bits::to_double(hi));
  // lo, lengthened by far more than its error, must not round hi + lo away from hi
  bool ok = __fadd_rn(hi, __fmul_rn(lo, 1.0001f)) == hi && (fabsf(hi) > 1e-30f || ra == 0.0);
  // S + sl = 1 - (hi + lo)^2
  const float p = __fmul_rn(hi, hi);
  const float pe = __fmaf_rn(__fmul_rn(2.f, hi), lo, __fmaf_rn(hi, hi, -p));
  const float sh = __fsub_rn(1.f, p);
  const float se = __fsub_rn(__fsub_rn(__fsub_rn(1.f, sh), p), pe);
  const float S = __fadd_rn(sh, se);
  const float sl = __fsub_rn(se, __fsub_rn(S, sh));
  ok = ok && S > 0.00390625f;
  // y = y0 + corr = (S + sl)^{-1/2}: one Newton step with the residual in pairs
  const float y0 = rsqrtf(S);
  const float q = __fmul_rn(y0, y0), qe = __fmaf_rn(y0, y0, -q);
  const float t = __fmul_rn(S, q);
  const float te = __fmaf_rn(sl, q, __fmaf_rn(S, qe, __fmaf_rn(S, q, -t)));
  const float d = __fsub_rn(__fsub_rn(1.f, t), te);
  const float corr = __fmul_rn(y0, __fmaf_rn(__fmul_rn(0.375f, d), d, __fmul_rn(0.5f, d)));
  const float k = __fmul_rn(y0, KAPPA);
  const float ke = __fmaf_rn(corr, KAPPA, __fmaf_rn(y0, KAPPA, -k));
  const float ch = __fadd_rn(k, ke);
  const float cl = __fsub_rn(ke, __fsub_rn(ch, k));
  const float err = __fmul_rn(ch, 0x1p-36f);
  ok = ok && __fadd_rn(ch, __fadd_rn(cl, err)) == ch && __fadd_rn(ch, __fsub_rn(cl, err)) == ch;
  float rho = hi, c = ch;
  if (!ok) {
    double r = cab / sqrt(C[(int64_t)a * m + a] * C[(int64_t)b * m + b]);
    if (!(1.0 - r * r >= DEGENERATE_1MR2)) {
      set_status(st, VL_ERR_DEGENERATE);
      r = 0.0;
    }
    rho = (float)r;
    c = (float)((double)KAPPA / sqrt(1.0 - r * r));
  }
  rho32[idx] = rho;
  c32[idx] = c;
}

// double-float accumulate (hi, lo) += x (TwoSum)
__device__ __forceinline__ void df_add(float& hi, float& lo, float x) {
  float s = hi + x;
  float bp = s - hi;
  float err = (hi - (s - bp)) + (x - bp);
  hi = s;
  lo += err;
}

// H of the residual of a on b from the split partials.
template <bool F32>
__device__ __forceinline__ double residual_entropy(const void* __restrict__ part_v, int64_t off,
                                                   int64_t mm, int splits, double inv_n) {
  if constexpr (F32) {
    // splits combined in double-float FP32 arithmetic, one FP64 sum per moment
    const float* p = static_cast<const float*>(part_v) + off;
    float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
#pragma unroll 4
    for (int s = 0; s < splits; ++s, p += 4 * mm) {
      df_add(h0, l0, p[0]);
      df_add(h0, l0, p[mm]);
      df_add(h1, l1, p[2 * mm]);
      df_add(h1, l1, p[3 * mm]);
    }
    const double s0 = bits::to_double(h0) + bits::to_double(l0);  // sum of log cosh u
    const double s1 = bits::to_double(h1) + bits::to_double(l1);  // sum of w e^{-u^2/2}
    return entropy_from_moments(s0 * inv_n, s1 * (inv_n * (LN2 / 2.0)));
  }
  const double* p = static_cast<const double*>(part_v) + off;
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
  for (int s = 0; s < splits; ++s, p += 2 * mm) {
    s0 += p[0];
    s1 += p[mm];
  }
  return entropy_from_moments(s0 * inv_n, s1 * inv_n);
}

// Hr and D = H(x_b) + H(r_a<-b) - H(x_a) - H(r_b<-a) from the partials and the
// variables' entropies hx.  One CTA per pair of FT x FT tiles mirrored at the
// diagonal: every entropy is computed once and exchanged through shared memory
// (not twice, once on each side of the diagonal), all global accesses run along
// rows, and the divisions by n are products.  FP64 instructions bound it (about 14
// an entry, 80 before): m = 400 13 us against 31, m = 1600 81 against 329.  Tiles of
// 8 keep the FP64 work of small m spread over enough SMs.
constexpr int FT = 8;
template <bool F32>
__global__ void __launch_bounds__(2 * FT * FT)
    measure_finalize_kernel(const void* __restrict__ part, int m, int splits, double inv_n,
                            const double* __restrict__ hx, double* __restrict__ Hx,
                            double* __restrict__ Hr, double* __restrict__ D) {
  pdl_begin(part, hx, Hx, Hr, D);
  __shared__ double hs[2][FT][FT + 1];
  int I, J;
  tile_coords(blockIdx.x, (m + FT - 1) / FT, I, J);
  // the first half of the threads takes the upper tile, the second the mirrored one
  const int side = threadIdx.x / (FT * FT), r = threadIdx.x / FT % FT, c = threadIdx.x % FT;
  const int a = (side ? J : I) * FT + r, b = (side ? I : J) * FT + c;
  const bool in = a < m && b < m && !(side && I == J);
  const int64_t off = (int64_t)a * m + b;
  double h = 0.0;
  if (in && a != b) h = residual_entropy<F32>(part, off, (int64_t)m * m, splits, inv_n);
  hs[side][r][c] = h;
  __syncthreads();
  if (!in) return;
  const double o = hs[I == J ? 0 : !side][c][r];  // H of the residual of b on a
  Hr[off] = h;
  D[off] = a == b ? 0.0 : hx[b] + h - hx[a] - o;
  if (Hx && a == b) Hx[a] = hx[a];
}

}  // namespace

// FP32 kernel configuration: micro-tile rows, samples per stage, CTAs per SM.
// 1 x 2 micro-tiles, 512 threads and one CTA per SM: measured at m = 400,
// n = 2500 against 2 x 2 micro-tiles with 256 threads (one or two CTAs per SM)
// and 64-192 sample stages, this was the fastest (148 vs 150-164 us).
constexpr int F32_MTI = 1;
constexpr int F32_TTS = 128;
constexpr int F32_MINB = 1;

// Sample splits for `slots` resident CTAs: the CTA count should fill whole
// waves (about 3-6 of them), each split at least two stages of `tts` long.
PairPlan plan_pairwise_slots(int m, int n, int slots, int tts, bool fp64, int num_sms) {
  PairPlan pl{};
  pl.m = m;
  pl.n = n;
  pl.m_pad = ((m + TB - 1) / TB) * TB;
  const int Tside = pl.m_pad / TB;
  pl.tiles = Tside * (Tside + 1) / 2;
  const int n_run = ((n + KRUN - 1) / KRUN) * KRUN;
  int max_split = std::max(1, n_run / (2 * tts));
  // a small problem that does not fill one wave even at this split count gets
  // shorter splits (down to 4 runs of samples each), up to one CTA per slot
  if ((long)pl.tiles * max_split < slots)
    max_split = std::max(max_split, std::min(n_run / (4 * KRUN), (slots + pl.tiles - 1) / pl.tiles));
  int splits = 1;
  double best = -1.0;
  for (int sp = 1; sp <= max_split; ++sp) {
    const long ctas = (long)pl.tiles * sp;
    const long waves = (ctas + slots - 1) / slots;
    if (waves > 8) break;
    const double eff = (double)ctas / (double)(waves * slots);
    // prefer full waves; among equals, at least 3 waves for load balance
    const double score = eff - (waves < 3 ? 0.05 * (3 - waves) : 0.0);
    if (score > best + 1e-9) {
      best = score;
      splits = sp;
    }
  }
  if (fp64) {
    // CTAs of FX_TH pairs, six to eight resident per SM: about four waves of
    // them so that the last one is short, splits of at least 16 samples, and
    // no more partials than vl_reserve counts
    const int pb = (int)(((int64_t)m * (m - 1) / 2 + FX_TH - 1) / FX_TH);
    const int64_t cap = 32 + 2048 * (int64_t)num_sms / ((int64_t)m * m);
    splits = (int)std::min<int64_t>({(24 * (int64_t)num_sms + pb - 1) / pb, cap,
                                     std::max(1, n_run / 16)});
    splits = std::max(1, splits);
  }
  int tps = (n_run + splits - 1) / splits;
  tps = ((tps + KRUN - 1) / KRUN) * KRUN;
  pl.splits = (n_run + tps - 1) / tps;
  pl.t_per_split = tps;
  pl.n_pad = ((n_run + 255) / 256) * 256;  // whole stages of any configuration
  return pl;
}

PairPlan plan_pairwise_split(int m, int n, int split_len) {
  PairPlan pl{};
  pl.m = m;
  pl.n = n;
  pl.m_pad = ((m + TB - 1) / TB) * TB;
  const int Tside = pl.m_pad / TB;
  pl.tiles = Tside * (Tside + 1) / 2;
  const int n_run = ((n + KRUN - 1) / KRUN) * KRUN;
  int tps = std::max(KRUN, ((std::min(split_len, n_run) + KRUN - 1) / KRUN) * KRUN);
  pl.splits = (n_run + tps - 1) / tps;
  tps = ((n_run + pl.splits - 1) / pl.splits + KRUN - 1) / KRUN * KRUN;  // even splits
  pl.splits = (n_run + tps - 1) / tps;
  pl.t_per_split = tps;
  pl.n_pad = ((n_run + 255) / 256) * 256;
  return pl;
}

PairPlan plan_pairwise(int m, int n, int num_sms, bool fp64) {
  return plan_pairwise_slots(m, n, F32_MINB * num_sms, F32_TTS, fp64, num_sms);
}

void launch_pair_consts(const double* C, const double* w, int m, float* rho32, float* c32,
                        int* st, Lane s) {
  int64_t tot = (int64_t)m * m;
  launch(pair_consts_kernel, (unsigned)((tot + 255) / 256), 256, 0, s, C, w, m, rho32, c32, st);
}

void launch_pair_consts64(const double* C, int m, double* rho64, double* c64, int* st,
                          Lane s) {
  int64_t tot = (int64_t)m * m;
  launch(pair_consts64_kernel, (unsigned)((tot + 255) / 256), 256, 0, s, C, m, rho64, c64, st);
}

template <int MTI, int TTS, int MINB>
void launch_pairwise_f32_cfg(const float* xt, const PairPlan& pl, const float* rho32,
                             const float* c32, float* part, Lane s) {
  const int n_run = ((pl.n + KRUN - 1) / KRUN) * KRUN;
  dim3 grid(pl.tiles, pl.splits);
  const size_t smem = sizeof(float) * 3 * TTS * 2 * TB;  // three stages of TTS x 64 samples
  static SmemOptIn opt;
  opt.allow(pairwise_f32_kernel<MTI, TTS, MINB>, smem);
  launch(pairwise_f32_kernel<MTI, TTS, MINB>, grid, TB / MTI * 16, smem, s, xt, pl.m, pl.m_pad,
         pl.m_pad / TB, n_run, pl.t_per_split, rho32, c32, part);
}

void launch_pairwise_f32(const float* xt, const PairPlan& pl, const float* rho32,
                         const float* c32, float* part, Lane s) {
  launch_pairwise_f32_cfg<F32_MTI, F32_TTS, F32_MINB>(xt, pl, rho32, c32, part, s);
}

PairJob make_pair_job(const float* xt, const PairPlan& pl, const float* rho32, const float* c32,
                      float* part) {
  PairJob j;
  j.xt = xt;
  j.rho32 = rho32;
  j.c32 = c32;
  j.part = part;
  j.m = pl.m;
  j.m_pad = pl.m_pad;
  j.T = pl.m_pad / TB;
  j.n_run = ((pl.n + KRUN - 1) / KRUN) * KRUN;
  j.tps = pl.t_per_split;
  return j;
}

void launch_pairwise_f32_list(const PairJob* jobs, const int4* items, int nitems, int grid,
                              Lane s) {
  constexpr int MTI = F32_MTI, TTS = F32_TTS, MINB = F32_MINB;
  const size_t smem = sizeof(float) * 3 * TTS * 2 * TB;
  static SmemOptIn opt;
  opt.allow(pairwise_f32_list_kernel<MTI, TTS, MINB>, smem);
  launch(pairwise_f32_list_kernel<MTI, TTS, MINB>, std::max(1, std::min(grid, nitems)), TB / MTI *
         16, smem, s, jobs, items, nitems);
}

void launch_pairwise_f64(const double* xt, const PairPlan& pl, const double* rho64,
                         const double* c64, double* part, Lane s) {
  const int64_t pairs = (int64_t)pl.m * (pl.m - 1) / 2;
  dim3 grid((unsigned)((pairs + FX_TH - 1) / FX_TH), pl.splits);
  launch(pairwise_f64_kernel, grid, FX_TH, 0, s, xt, pl.m, pl.m_pad, pl.n, pl.t_per_split, rho64,
         c64, part);
}

void launch_measure_finalize(const void* part, const PairPlan& pl, const double* hx, double* Hx,
                             double* Hr, double* D, bool fp32_parts, Lane s) {
  const unsigned T = (pl.m + FT - 1) / FT;
  launch(fp32_parts ? measure_finalize_kernel<true> : measure_finalize_kernel<false>, T * (T + 1) /
         2, 2 * FT * FT, 0, s, part, pl.m, pl.splits, 1.0 / pl.n, hx, Hx, Hr, D);
}

}  // namespace vl
