// Cholesky factorisation A = L L^T of an FP32 SPD matrix by one thread-block
// cluster: the normal-equation matrix of the VAR fit (Sec. 4.1) and the
// causally ordered residual covariance whose factor gives B0 (Sec. 4.2 item 5)
// are both factored here on the mixed-precision path.
//
// GB300 design.  The matrix is far too small to fill the GPU: what bounds it is
// the chain of diagonal blocks, each factor needing the panel and the update of
// the one before.  So one CTA of the cluster (rank 0, the chain) does nothing
// but that chain, entirely in its own shared memory, and the others (the
// workers) hold the rest of the lower triangle, dealt by 32-row blocks, and
// keep everything further from the diagonal up to date.  Period p of the chain:
//   - warps 0 and 1 factor and invert diagonal block p;
//   - meanwhile the other ten warps take row block I = p + 1 over from its
//     worker (tiles I-3 .. I), apply to it the block columns I-3 and I-2 (whose
//     panels the chain holds or forms), and store what has become final;
//   - then all warps form L[p+1][p] and apply it to diagonal block p + 1.
// Period p of a worker, for its row blocks I >= p + 2: block column p - 2 is
// applied to the tiles J >= p - 1, then L[I][p-1] is formed with the inverse
// that the chain finished in the period before.  So a result has a whole period
// on its way between CTAs, and one cluster barrier per period (arrive and wait
// apart) orders it all.  All diagonal blocks are factored on one SM, whose
// instruction cache keeps that long straight-line code.
//
// What crosses CTAs goes through L2: every finished tile of L and every inverse
// is also written to a global scratch as a packed 4 KB tile (float4 q4 of row r
// at q4 32 + r, so that a warp whose lane holds a row reads it coalesced).
// Distributed shared memory was tried for it: it moves about 8 bytes a clock out
// of one SM here, and seven workers reading the chain's tiles made a period
// 25,000 clocks.
//
// Measured, n = 400, a launch in a stream of calls: 90 us, against 145-150 us with
// the row blocks dealt round-robin and every block column's inverse and panels
// crossing the cluster inside the chain (under the profiler, caches cold, 94 and
// 170; 32-row blocks and the order of every sum are the same: the
// factors are bit-identical).
//
// Cluster size: one worker for each row block below the third, up to seven (the
// portable cluster of 8 CTAs).
//
// Outputs: L in the lower triangle of A (the strict upper triangle is left as
// it was) and, per 64-block of rows, the inverse of the 64 x 64 diagonal block
// of L (dinv), built from the two 32 x 32 inverses as
// [A 0; B C]^{-1} = [A^{-1} 0; -C^{-1} B A^{-1}  C^{-1}].
// A pivot at or below rel_tol * (its original diagonal) sets VL_ERR_RANK.
#include <algorithm>

#include "vl_internal.cuh"

namespace vl {

namespace {

constexpr int CB = 32;        // block column width
constexpr int RS = CB + 4;    // shared row stride: 16-byte rows, conflict-free float4 columns
constexpr int TILE = CB * RS; // floats of one 32 x 32 tile in the chain's memory
constexpr int CTH = 384;      // threads per CTA
constexpr int NWARP = CTH / 32;
constexpr int SHADOW = NWARP - 2;  // the chain's warps beside the factoring two
constexpr int CL_MAX = 8;           // CTAs per cluster (portable maximum)
constexpr int CL_NMAX = 512;        // largest n handled
constexpr int BMAX = CL_NMAX / CB;  // most row blocks

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Global scratch of a factorisation with workers: packed tiles of L (I, k), the
// packed inverses, and per row block the three tiles its worker hands to the
// chain (row-major).
struct Scratch {
  float *L, *inv, *hand;
  __device__ float* tile(int I, int k) const { return L + (size_t)(I * (I + 1) / 2 + k) * CB * CB; }
  __device__ float* inverse(int k) const { return inv + (size_t)k * CB * CB; }
  __device__ float* handed(int I, int J) const {  // I-2 <= J <= I
    return hand + (size_t)(3 * I + J - I + 2) * CB * CB;
  }
};
size_t scratch_floats(int nblk) {
  return (size_t)(nblk * (nblk + 1) / 2 + 4 * nblk) * CB * CB;
}

// The chain's shared memory (floats): rows 0 .. 3 of a ring (row block I in
// slot I mod 4), each the tiles (I, I-3) .. (I, I) at 32 x RS; the inverses of
// the last four diagonal blocks; scratch of the factor and of the 64-blocks.
constexpr int RING = 4;
__host__ __device__ constexpr int ch_tile(int I, int J) {  // tile (I, J), I-3 <= J <= I
  return ((I % RING) * 4 + (J - I + 3)) * TILE;
}
__host__ __device__ constexpr int ch_inv(int k) { return (RING * 4 + k % RING) * TILE; }
constexpr int CH_COL = (RING * 5) * TILE;  // the factor's columns, one tile
constexpr int CH_FLOATS = CH_COL + TILE;

// A worker's row block b: 32 rows of ldb(b) floats, columns 0 .. 32(b+1)-1.
__host__ __device__ constexpr int ldb(int b) { return CB * (b + 1) + 4; }
// Row blocks 3 .. nblk-1 dealt, longest first, back and forth over W workers:
// the owner's rank of block b.
__host__ __device__ inline int row_owner(int b, int nblk, int W) {
  const int q = nblk - 1 - b, round = q / W, at = q % W;
  return 1 + ((round & 1) ? W - 1 - at : at);
}
// Offset (floats) of block b in its owner's memory: after the longer ones.
inline int row_off(int b, int nblk, int W) {
  int o = 0;
  for (int c = nblk - 1; c > b; --c)
    if (row_owner(c, nblk, W) == row_owner(b, nblk, W)) o += CB * ldb(c);
  return o;
}

// Warps 0 and 1: warp 0 factors the 32 x 32 block (rows of stride RS, nb valid)
// in place, warp 1 builds L^{-1} into li behind it, from the columns warp 0
// leaves in col (row j of stride RS: the multipliers of rows j + 1 .. 31, then
// zeros; at 32 the threshold of pivot j + 1, at 34 1 / L[j][j], at 35 L[j][j]).
// Every four columns warp 0 arrives, without waiting, at one of the named barriers
// 5 .. 12, each used once per block.
//
// Lane r holds row r from column j on, a[c] = entry (r, j + c): the update writes
// entry c + 1 into register c, so that the steps of a group of eight are the same
// code (W registers wide, W = 32, 24, 16, 8) and stay a loop.  Unrolled over all
// columns (two times 30 KB of straight-line code), a block took 5,000 to 9,700
// clocks, waiting for instructions.  A step's chain is a product, the next pivot,
// a shuffle and a reciprocal root; the multipliers' way through shared memory
// runs beside the last two.
template <int W>
__device__ __forceinline__ void factor_steps(float (&a)[CB], float& rs, float& dg, bool& lbad,
                                             int nb, float* col) {
  const int lane = threadIdx.x & 31;
#pragma unroll 2
  for (int j = CB - W; j < CB - W + 8; ++j) {
    float* cj = col + j * RS;
    const float tj = cj[CB];  // the next pivot's threshold
    const float l = lane > j ? a[0] * rs : 0.f;
    const float piv = fmaf(-l, l, a[1]);
    float d;  // before the shared-memory traffic, which would queue in front of it
    asm volatile("shfl.sync.idx.b32 %0, %1, %2, 31, 0xffffffff;"
                 : "=f"(d)
                 : "f"(piv), "r"(j + 1)
                 : "memory");
    cj[(lane - j - 1) & 31] = l;
    if (lane == 0) *reinterpret_cast<float2*>(cj + CB + 2) = make_float2(rs, dg);
    __syncwarp();
    float4 v[W / 4];
#pragma unroll
    for (int c = 0; c < W / 4; ++c) v[c] = *reinterpret_cast<const float4*>(cj + 4 * c);
    const bool ok = d > tj;
    lbad |= !ok && j + 1 < nb;
    const float dd = ok ? d : 1.f;
    rs = rsqrtf(dd);
    dg = dd * rs;
    if ((j & 3) == 3) asm volatile("bar.arrive %0, 64;" ::"r"(5 + (j >> 2)) : "memory");
#pragma unroll
    for (int c = 0; c < W / 4; ++c) {
      a[4 * c] = fmaf(-l, v[c].x, a[4 * c + 1]);
      a[4 * c + 1] = fmaf(-l, v[c].y, a[4 * c + 2]);
      a[4 * c + 2] = fmaf(-l, v[c].z, a[4 * c + 3]);
      a[4 * c + 3] = 4 * c + 4 < W ? fmaf(-l, v[c].w, a[(4 * c + 4) % CB]) : 0.f;
    }
  }
}
// Lane c holds column c of L^{-1}: s[i] = sum_{q < j} L[j + i][q] x_q.
template <int W>
__device__ __forceinline__ void inverse_steps(float (&s)[CB], float* li, const float* col) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int j0 = CB - W; j0 < CB - W + 8; j0 += 4) {
    asm volatile("bar.sync %0, 64;" ::"r"(5 + (j0 >> 2)) : "memory");
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = j0 + e;
      const float* cj = col + j * RS;
      const float x = ((lane == j ? 1.f : 0.f) - s[0]) * cj[CB + 2];
      li[j * RS + lane] = x;
#pragma unroll
      for (int c = 0; c < W / 4; ++c) {
        const float4 v = *reinterpret_cast<const float4*>(cj + 4 * c);
        s[4 * c] = fmaf(v.x, x, s[4 * c + 1]);
        s[4 * c + 1] = fmaf(v.y, x, s[4 * c + 2]);
        s[4 * c + 2] = fmaf(v.z, x, s[4 * c + 3]);
        s[4 * c + 3] = 4 * c + 4 < W ? fmaf(v.w, x, s[(4 * c + 4) % CB]) : 0.f;
      }
    }
  }
}

// L from its columns, rows of stride RS; warps w of nw.
__device__ __forceinline__ void write_factor(float* blk, const float* col, int w, int nw) {
  const int r = threadIdx.x & 31;
  for (int c = w; c < CB; c += nw)
    if (c <= r) blk[r * RS + c] = col[c * RS + (c == r ? CB + 3 : r - c - 1)];
}

__device__ __noinline__ bool factor_invert2(const float* blk, int nb, const double* diag0k,
                                            float rel_tol, float* li, float* col) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned full = 0xffffffffu;
  bool lbad = false;
  if (warp == 0) {
    float a[CB];
#pragma unroll
    for (int c4 = 0; c4 < CB; c4 += 4) {
      const float4 v = *reinterpret_cast<const float4*>(blk + lane * RS + c4);
      a[c4] = v.x;
      a[c4 + 1] = v.y;
      a[c4 + 2] = v.z;
      a[c4 + 3] = v.w;
    }
#pragma unroll
    for (int c = 0; c < CB; ++c)
      if (!(lane < nb && c < nb && c <= lane)) a[c] = (c == lane) ? 1.f : 0.f;
    const float thr = lane < nb ? (float)(rel_tol * diag0k[lane]) : 0.f;
    col[((lane - 1) & 31) * RS + CB] = thr;
    __syncwarp();
    const float d = __shfl_sync(full, a[0], 0);
    const bool ok = d > __shfl_sync(full, thr, 0);
    lbad = !ok;
    const float dd = ok ? d : 1.f;
    float rs = rsqrtf(dd), dg = dd * rs;
    factor_steps<32>(a, rs, dg, lbad, nb, col);
    factor_steps<24>(a, rs, dg, lbad, nb, col);
    factor_steps<16>(a, rs, dg, lbad, nb, col);
    factor_steps<8>(a, rs, dg, lbad, nb, col);
  } else {
    float s[CB];
#pragma unroll
    for (int i = 0; i < CB; ++i) s[i] = 0.f;
    inverse_steps<32>(s, li, col);
    inverse_steps<24>(s, li, col);
    inverse_steps<16>(s, li, col);
    inverse_steps<8>(s, li, col);
  }
  __syncwarp();
  return __any_sync(full, lbad);
}

// Tile products of one warp.  Lane (ry, cx) = (lane % 8, lane / 8) accumulates
// the entries (ry + 8 u, cx + 4 k), u < U, k < K, of X Y^T, q ascending over the
// first 4 nq columns: (U + K) vector loads from shared memory feed 4 U K
// multiply-adds.  Shared memory returns 128 bytes a clock to an SM whatever the
// lanes share, so a product of one row per step with broadcast rows (U + K = 1
// load for 4 multiply-adds) spends four times the arithmetic's time on them.
// Rows ry and ry + 8, and columns cx .. cx + 3, fall into distinct banks for
// row strides of 4 mod 32 floats.
template <int U, int K>
__device__ __forceinline__ void tile_dots(float (&acc)[U][K], const float* X, int ldx,
                                          const float* Y, int nq) {
  const int ry = threadIdx.x & 7, cx = (threadIdx.x >> 3) & 3;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int k = 0; k < K; ++k) acc[u][k] = 0.f;
#pragma unroll 2
  for (int q4 = 0; q4 < nq; ++q4) {
    float4 x[U], y[K];
#pragma unroll
    for (int u = 0; u < U; ++u)
      x[u] = *reinterpret_cast<const float4*>(X + (ry + 8 * u) * ldx + 4 * q4);
#pragma unroll
    for (int k = 0; k < K; ++k)
      y[k] = *reinterpret_cast<const float4*>(Y + (cx + 4 * k) * RS + 4 * q4);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[u][k] = fmaf(x[u].x, y[k].x, acc[u][k]);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[u][k] = fmaf(x[u].y, y[k].y, acc[u][k]);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[u][k] = fmaf(x[u].z, y[k].z, acc[u][k]);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[u][k] = fmaf(x[u].w, y[k].w, acc[u][k]);
  }
}

// out -= P Q^T on 8 U rows and 4 K columns (out, P and Q already at the first
// row or column of the part); Q rows of stride RS.  G (optional): the result
// also to a row-major 32-wide tile.
template <int U, int K>
__device__ __noinline__ void update_part(float* out, int ldo, const float* P, int ldp,
                                         const float* Q, float* G) {
  const int ry = threadIdx.x & 7, cx = (threadIdx.x >> 3) & 3;
  float acc[U][K];
  tile_dots<U, K>(acc, P, ldp, Q, CB / 4);
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int r = ry + 8 * u, c = cx + 4 * k;
      const float v = out[r * ldo + c] - acc[u][k];
      out[r * ldo + c] = v;
      if (G) G[r * CB + c] = v;
    }
}

// X <- X inv^T in place on 8 U rows, all 32 columns (inv lower triangular: the
// first 16 columns stop at q = 15, adding zeros would change nothing).
template <int U>
__device__ __noinline__ void panel_part(float* X, int ldx, const float* inv) {
  const int ry = threadIdx.x & 7, cx = (threadIdx.x >> 3) & 3;
  float lo[U][4], hi[U][4];
  tile_dots<U, 4>(lo, X, ldx, inv, CB / 8);
  tile_dots<U, 4>(hi, X, ldx, inv + 16 * RS, CB / 4);
  __syncwarp();
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      X[(ry + 8 * u) * ldx + cx + 4 * k] = lo[u][k];
      X[(ry + 8 * u) * ldx + 16 + cx + 4 * k] = hi[u][k];
    }
  __syncwarp();
}

// The same for a whole tile of the chain by four warps (w = 0 .. 3: a half of the
// rows by a half of the columns each), which wait for one another at named
// barrier `bar` between reading X and writing it.
__device__ __noinline__ void panel_quarter(float* X, const float* inv, int w, int bar) {
  const int ry = threadIdx.x & 7, cx = (threadIdx.x >> 3) & 3;
  X += (w >> 1) * 16 * RS;
  float acc[2][4];
  tile_dots<2, 4>(acc, X, RS, inv + (w & 1) * 16 * RS, (w & 1) ? CB / 4 : CB / 8);
  asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int k = 0; k < 4; ++k) X[(ry + 8 * u) * RS + (w & 1) * 16 + cx + 4 * k] = acc[u][k];
}

// One warp packs float4 columns 2 part, 2 part + 1 (part = 0 .. 3) of a tile,
// rows r0 .. r0 + 31.
__device__ __forceinline__ void pack_part(float* dst, const float* tile, int ld, int part) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q4 = 2 * part; q4 < 2 * part + 2; ++q4)
    reinterpret_cast<float4*>(dst)[q4 * CB + lane] =
        *reinterpret_cast<const float4*>(tile + lane * ld + 4 * q4);
}
// float4 e (0 .. 255) of a packed tile, to its place in a tile of stride RS
__device__ __forceinline__ float4* unpack_at(float* tile, int e) {
  return reinterpret_cast<float4*>(tile + (e % CB) * RS + 4 * (e / CB));
}

__device__ __forceinline__ void shadow_sync() {
  asm volatile("bar.sync 4, %0;" ::"n"(SHADOW * 32) : "memory");
}

// Lower-left quadrant -C^{-1} (B A^{-1}) of a 64-block's inverse: step 0 B
// A^{-1} into t, step 1 the product with -C^{-1} to out; rows r0 .. r0 + 3, all
// tiles at stride RS.
__device__ __noinline__ void combine_step(const float* B, const float* ai, const float* ci,
                                          float* t, float* out, int step, int r0) {
  const int lane = threadIdx.x & 31;
  const float* X = step ? ci : B;
  const float* Y = step ? t : ai;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
  for (int q = 0; q < CB; ++q) {
    const float y = Y[q * RS + lane];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float x = X[(r0 + u) * RS + q];
      acc[u] = fmaf(step ? -x : x, y, acc[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (step)
      out[(CB + r0 + u) * CHOL_NB + lane] = acc[u];
    else
      t[(r0 + u) * RS + lane] = acc[u];
  }
}

// One CTA: the 64-block b of dinv from the two inverses ai, ci and the tile B
// between them (ci, B unused if the second row block does not exist), all in
// shared memory at stride RS; t a scratch tile there.
__device__ void emit_inverse(const float* ai, const float* ci, const float* B, float* t,
                             float* __restrict__ dinv, int b, bool pair) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* out = dinv + (size_t)b * CHOL_NB * CHOL_NB;
  for (int a = warp; a < CB; a += NWARP) {
    out[a * CHOL_NB + lane] = ai[a * RS + lane];
    out[a * CHOL_NB + CB + lane] = 0.f;
    out[(CB + a) * CHOL_NB + CB + lane] = pair ? ci[a * RS + lane] : (a == lane ? 1.f : 0.f);
    if (!pair) out[(CB + a) * CHOL_NB + lane] = 0.f;
  }
  if (!pair) return;
  if (warp < 8) combine_step(B, ai, ci, t, out, 0, warp * 4);
  __syncthreads();
  if (warp < 8) combine_step(B, ai, ci, t, out, 1, warp * 4);
}

__device__ void chain_cta(float* sm, float* __restrict__ A, int64_t lda, int n, int nblk,
                          Scratch S, float* __restrict__ dinv, const double* __restrict__ diag0,
                          float rel_tol, int* st) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool workers = nblk > 3;
  bool bad = false;
  // row blocks 0 .. 3 (zeros beyond n; of row block 3 the tiles 1 .. 3)
  for (int t = warp; t < min(4, nblk) * 3 * CB; t += NWARP) {
    const int I = t / (3 * CB), J = (t / CB) % 3 + (I == 3), a = t % CB;
    const int g = I * CB + a, gc = J * CB + lane;
    if (J <= I)
      sm[ch_tile(I, J) + a * RS + lane] = (g < n && gc < n) ? A[(int64_t)g * lda + gc] : 0.f;
  }
  __syncthreads();
  cluster_arrive();
  for (int p = 0; p < nblk; ++p) {
    const int I = p + 1;
    if (warp < 2) {
      bad |= factor_invert2(sm + ch_tile(p, p), min(CB, n - p * CB), diag0 + p * CB, rel_tol,
                            sm + ch_inv(p), sm + CH_COL);
      cluster_wait();
    } else {
      const int sw = warp - 2;
      cluster_wait();  // the workers' period p - 1
      if (I < nblk && I >= 3) {
        // take row block I over: the packed tile (I, I-3), and the three handed
        // ones (row block 3's are here already); 256 float4 each
        float4 v[4];
        const int cnt = (I == 3 ? 1 : 4) * (CB * CB / 4);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int x = tid - 64 + u * SHADOW * 32, J = I - 3 + x / (CB * CB / 4);
          if (x < cnt)
            v[u] = __ldcg(reinterpret_cast<const float4*>(J == I - 3 ? S.tile(I, J)
                                                                     : S.handed(I, J)) +
                          x % (CB * CB / 4));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int x = tid - 64 + u * SHADOW * 32, J = I - 3 + x / (CB * CB / 4);
          const int e = x % (CB * CB / 4);
          if (x < cnt)
            *(J == I - 3 ? unpack_at(sm + ch_tile(I, J), e)
                         : reinterpret_cast<float4*>(sm + ch_tile(I, J) + e / 8 * RS) + e % 8) =
                v[u];
        }
        shadow_sync();
        // block column I-3 on the tiles (I, I-2) .. (I, I)
        if (sw < 6) {
          const int J = I - 2 + (sw >> 1), c = (sw & 1) * 16;
          update_part<4, 4>(sm + ch_tile(I, J) + c, RS, sm + ch_tile(I, I - 3), RS,
                            sm + ch_tile(J, I - 3) + c * RS, nullptr);
        }
        shadow_sync();
      }
      if (I < nblk && I >= 2) {
        if (sw < 4) panel_quarter(sm + ch_tile(I, I - 2), sm + ch_inv(I - 2), sw, 13);
        shadow_sync();
        // block column I-2 on the tiles (I, I-1), (I, I)
        if (sw < 4) {
          const int J = I - 1 + (sw >> 1), c = (sw & 1) * 16;
          update_part<4, 4>(sm + ch_tile(I, J) + c, RS, sm + ch_tile(I, I - 2), RS,
                            sm + ch_tile(J, I - 2) + c * RS, nullptr);
        } else if (sw < 8 && workers) {
          pack_part(S.tile(I, I - 2), sm + ch_tile(I, I - 2), RS, sw - 4);
        }
      }
    }
    __syncthreads();
    if (warp >= 8) {
      write_factor(sm + ch_tile(p, p), sm + CH_COL, warp - 8, 4);
      if (workers) {
        pack_part(S.inverse(p), sm + ch_inv(p), RS, warp - 8);
        asm volatile("bar.sync 14, 128;" ::: "memory");
        pack_part(S.tile(p, p), sm + ch_tile(p, p), RS, warp - 8);
      }
    }
    if (I < nblk) {
      if (warp < 4) panel_quarter(sm + ch_tile(I, p), sm + ch_inv(p), warp, 13);
      __syncthreads();
      if (warp < 4) {  // the lower triangle: quarters (0, 0), (1, 0) and (1, 1)
        const int o = (warp >> 1) * 16, c = (warp & 1) * 16;
        if (c <= o)
          update_part<2, 4>(sm + ch_tile(I, I) + o * RS + c, RS, sm + ch_tile(I, p) + o * RS, RS,
                            sm + ch_tile(I, p) + c * RS, nullptr);
      } else if (warp >= 8 && workers) {
        pack_part(S.tile(I, p), sm + ch_tile(I, p), RS, warp - 8);
      }
      __syncthreads();
    }
    cluster_arrive();
  }
  cluster_wait();
  if (bad && tid == 0) set_status(st, VL_ERR_RANK);
  if (workers) return;
  // alone: everything is still in the ring
  __syncthreads();
  for (int t = warp; t < nblk * nblk * CB; t += NWARP) {
    const int I = t / CB / nblk, J = t / CB % nblk, a = t % CB;
    const int g = I * CB + a, gc = J * CB + lane;
    if (J <= I && g < n && gc <= g) A[(int64_t)g * lda + gc] = sm[ch_tile(I, J) + a * RS + lane];
  }
  for (int b = 0; 2 * b < nblk; ++b)
    emit_inverse(sm + ch_inv(2 * b), sm + ch_inv(2 * b + 1), sm + ch_tile(2 * b + 1, 2 * b),
                 sm + CH_COL, dinv, b, 2 * b + 1 < nblk);
}

__device__ void worker_cta(float* sm, float* __restrict__ A, int64_t lda, int n, int nblk, int W,
                           Scratch S, float* __restrict__ dinv, int rank, int own) {
  __shared__ int mine[BMAX];  // this worker's row blocks, longest first
  __shared__ int off[BMAX];   // and their offsets
  __shared__ int nmine;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // staged tiles: the inverse, L[p-1][p-2], then L[J][p-2] for J >= p
  float* stage = sm + own;
  if (tid == 0) {
    int c = 0, o = 0;
    for (int b = nblk - 1; b >= 3; --b)
      if (row_owner(b, nblk, W) == rank) {
        mine[c] = b;
        off[c++] = o;
        o += CB * ldb(b);
      }
    nmine = c;
  }
  __syncthreads();
  const int nm = nmine;
  // owned row blocks (zeros beyond n), one row per warp and turn
  for (int t = warp; t < nm * CB; t += NWARP) {
    const int b = mine[t / CB], a = t % CB, g = b * CB + a, w = CB * (b + 1);
    float* dst = sm + off[t / CB] + a * ldb(b);
    const float* src = A + (int64_t)g * lda;
    for (int c = lane; c < w; c += 8 * 32) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int cc = c + 32 * u;
        v[u] = (cc < w && g < n && cc < n) ? src[cc] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (c + 32 * u < w) dst[c + 32 * u] = v[u];
    }
  }
  __syncthreads();
  cluster_arrive();
  for (int p = 0; p < nblk; ++p) {
    cluster_wait();  // period p - 1 of every CTA
    int act = 0;     // this worker's row blocks I >= p + 2 (the first of `mine`)
    while (act < nm && mine[act] >= p + 2) ++act;
    if (p >= 1 && act) {
      const int staged = 2 + (p >= 2 ? mine[0] + 1 - p : 0);
      for (int x0 = tid; x0 < staged * (CB * CB / 4); x0 += 4 * CTH) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int x = x0 + u * CTH, i = x / (CB * CB / 4), e = x % (CB * CB / 4);
          if (i >= staged || (i == 1 && p < 2)) continue;
          const float* src = i == 0 ? S.inverse(p - 1) : S.tile(p - 2 + i, p - 2);
          v[u] = __ldcg(reinterpret_cast<const float4*>(src) + e);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int x = x0 + u * CTH, i = x / (CB * CB / 4), e = x % (CB * CB / 4);
          if (i >= staged || (i == 1 && p < 2)) continue;
          *unpack_at(stage + i * TILE, e) = v[u];
        }
      }
      __syncthreads();
      // the tiles (I, p-1): block column p-2, then the panel with the inverse;
      // 16 rows a warp
      for (int t = warp; t < 2 * act; t += NWARP) {
        const int ld = ldb(mine[t >> 1]), o = (t & 1) * 16 * ld;
        float* X = sm + off[t >> 1] + o + (p - 1) * CB;
        if (p >= 2) update_part<2, 8>(X, ld, X - CB, ld, stage + TILE, nullptr);
        __syncwarp();
        panel_part<2>(X, ld, stage);
      }
      // block column p-2 on the tiles J = p .. I of every row block, a tile a
      // warp; row block p + 2, which the chain takes over in the next period,
      // goes to global memory as well
      int tasks = 0;
      for (int a = 0; p >= 2 && a < act; ++a) tasks += mine[a] + 1 - p;
      for (int t = (warp + NWARP - 2 * act % NWARP) % NWARP; t < tasks; t += NWARP) {
        int a = 0, x = t;
        while (x >= mine[a] + 1 - p) x -= mine[a++] + 1 - p;
        const int I = mine[a], J = p + x, ld = ldb(I);
        float* row = sm + off[a];
        update_part<4, 8>(row + J * CB, ld, row + (p - 2) * CB, ld, stage + (2 + x) * TILE,
                          I == p + 2 ? S.handed(I, J) : nullptr);
      }
    }
    __syncthreads();
    if (p >= 1)  // publish the panel tiles
      for (int t = warp; t < 4 * act; t += NWARP)
        pack_part(S.tile(mine[t >> 2], p - 1), sm + off[t >> 2] + (p - 1) * CB,
                  ldb(mine[t >> 2]), t & 3);
    cluster_arrive();
  }
  cluster_wait();
  // the factor to A: the own row blocks from shared memory up to tile I-3, the
  // chain's tiles (I, I-2) .. (I, I) from the scratch
  for (int t = warp; t < nm * CB; t += NWARP) {
    const int b = mine[t / CB], a = t % CB, g = b * CB + a;
    const float* src = sm + off[t / CB] + a * ldb(b);
    if (g < n)
      for (int c = lane; c < CB * (b - 2); c += 32) A[(int64_t)g * lda + c] = src[c];
  }
  for (int t = (rank - 1) * NWARP + warp; t < 3 * nblk * CB; t += W * NWARP) {
    const int I = t / (3 * CB), J = I - 2 + t / CB % 3, a = t % CB;
    const int g = I * CB + a, gc = J * CB + lane;
    if (J >= 0 && g < n && gc <= g)
      A[(int64_t)g * lda + gc] = __ldcg(S.tile(I, J) + (lane >> 2) * 4 * CB + a * 4 + (lane & 3));
  }
  // and the inverses, a 64-block a worker and turn
  __syncthreads();
  for (int b = rank - 1; 2 * b < nblk; b += W) {
    const bool pair = 2 * b + 1 < nblk;
    for (int x = tid; x < (pair ? 3 : 1) * (CB * CB / 4); x += CTH) {
      const int i = x / (CB * CB / 4), e = x % (CB * CB / 4);
      const float* src = i == 2 ? S.tile(2 * b + 1, 2 * b) : S.inverse(2 * b + i);
      *unpack_at(sm + i * TILE, e) = __ldcg(reinterpret_cast<const float4*>(src) + e);
    }
    __syncthreads();
    emit_inverse(sm, sm + TILE, sm + 2 * TILE, sm + 3 * TILE, dinv, b, pair);
    __syncthreads();
  }
}

// One cluster factors A in place.
__global__ void __launch_bounds__(CTH, 1)
    chol_cluster_kernel(float* __restrict__ A, int64_t lda, int n, float* __restrict__ dinv,
                        const double* __restrict__ diag0, float rel_tol, float* scratch, int own,
                        int* st) {
  pdl_wait(diag0);  // all else is written here too
  extern __shared__ __align__(16) float cc_smem[];
  const int nblk = (n + CB - 1) / CB, W = (int)cluster_size() - 1, rank = (int)cluster_rank();
  const size_t tiles = (size_t)(nblk * (nblk + 1) / 2) * CB * CB;
  const Scratch S{scratch, scratch + tiles, scratch + tiles + (size_t)nblk * CB * CB};
  if (rank == 0)
    chain_cta(cc_smem, A, lda, n, nblk, S, dinv, diag0, rel_tol, st);
  else
    worker_cta(cc_smem, A, lda, n, nblk, W, S, dinv, rank, own);
}

// The cluster for n: its CTAs, the floats of a worker's row blocks and the
// shared memory of each CTA (n = 512: 190 KB).
struct Shape {
  int cl, own;
  size_t smem;
};
Shape cluster_shape(int n) {
  const int nblk = (n + CB - 1) / CB;
  Shape h{};
  h.cl = std::min(CL_MAX, 1 + std::max(0, nblk - 3));
  for (int b = 3; b < nblk; ++b)
    h.own = std::max(h.own, row_off(b, nblk, h.cl - 1) + CB * ldb(b));
  h.smem = sizeof(float) * (size_t)std::max(CH_FLOATS, h.cl > 1 ? h.own + (2 + nblk) * TILE : 0);
  return h;
}

}  // namespace

// Launch the cluster factorisation; false if n is out of range, the scratch too
// small or the cluster not launched (the caller then uses another path).
bool launch_chol_cluster(float* A, int64_t lda, int n, float* dinv, const double* diag0,
                         float rel_tol, float* scratch, size_t scratch_cap, int* st,
                         Lane s) {
  if (n < 1 || n > CL_NMAX) return false;
  const int nblk = (n + CB - 1) / CB;
  if (nblk > 3 && scratch_floats(nblk) > scratch_cap) return false;
  const Shape h = cluster_shape(n);
  static SmemOptIn smem;
  if (!smem.allow(chol_cluster_kernel, cluster_shape(CL_NMAX).smem)) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(h.cl, 1, 1);
  cfg.blockDim = dim3(CTH, 1, 1);
  cfg.dynamicSmemBytes = h.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = h.cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  at[1] = pdl_attribute();
  cfg.numAttrs = s.overlap ? 2 : 1;
  note_launch();
  if (cudaLaunchKernelEx(&cfg, chol_cluster_kernel, A, lda, n, dinv, diag0, rel_tol, scratch,
                         h.own, st) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

}  // namespace vl
