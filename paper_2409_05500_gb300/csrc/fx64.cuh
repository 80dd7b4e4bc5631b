// Fixed-point evaluation of the two per-sample entropy functions for the FP64
// measure, and exact sums of them.
//
// This part issues FP64 at 1.6 operations per clock per SM, so CUDA's FP64 exp
// and log1p cost ~50 SM clocks a sample; the 32-bit integer multiplier runs at
// 30 to 60 times that rate.  Here a sample enters as the FP64 value
// w = kappa u (kappa = 2 log2 e) and from there on everything is 63-bit
// fixed-point integer arithmetic:
//     |w|                      units of 2^-57
//     log1p(e^{-2|u|})         = log1p(2^{-|w|}), units of 2^-63
//     kappa u e^{-u^2/2}       = w 2^{-w^2 ln2 / 8}, units of 2^-57
// the first within a unit of 2^-57, the second within a few of 2^-58, and the third,
// whose exponent w^2 ln2 / 8 is cut to units of 2^-54, so that u e^{-u^2/2} is within
// 7e-17 (3.2e-17 the largest seen; all checked against extended precision on the
// CPU): below FP64's own rounding of the same functions, 1.1e-16.  The sums over the
// samples are exact 96-bit integers.  The result is therefore closer to the exact
// moments than sums of FP64 functions are.
//
// 2^{-z}: z = n + j / 1024 + r, the table value 2^{-j/1024} and a degree-4
// series in r < 2^-10.  log1p(y): (1 + y) R_j = 1 + t with the 16-bit
// reciprocal R_j = ceil(2^16 / (1 + j / 256)), j the top eight bits of y, so
// that 0 <= t < 2^-7.9; -ln(R_j / 2^16) from a table and the series of
// log1p(t) to t^7.  Every series is evaluated by Horner's rule with each stage
// only as wide as its weight in the result needs: 32-bit products for the high
// powers, 64-bit ones for the low.
#pragma once

#include <cuda_runtime.h>

namespace vl {
namespace fx {

typedef unsigned long long u64;
typedef unsigned int u32;

// 2^{-a/32} and 2^{-a/1024} in units of 2^-63 (the kernels multiply them into
// a table of 2^{-j/1024} in shared memory); -ln(R_j / 2^16) in units of 2^-63.
static __constant__ unsigned long long kExpHi[32] = {
    0x7fffffffffffffffull, 0x7d41d96db915019dull, 0x7a92be8a92436616ull, 0x77f25ccdee6d7ae6ull,
    0x75606373ee921c97ull, 0x72dc8373be41a454ull, 0x70666f76154a7089ull, 0x6dfddbcbed791babull,
    0x6ba27e656b4eb57aull, 0x69540ec8f895722dull, 0x6712460a8fc24072ull, 0x64dcdec3371793d1ull,
    0x62b39508aa836d6full, 0x6096266533384a2bull, 0x5e8451cfac061b5full, 0x5c7dd7a3b17dcf75ull,
    0x5a827999fcef3242ull, 0x5891fac0e95612c8ull, 0x56ac1f752150a563ull, 0x54d0ad5a753e077cull,
    0x52ff6b54d8a89c75ull, 0x513821818624b40cull, 0x4f7a993048d088d7ull, 0x4dc69cdceaa72a9cull,
    0x4c1bf828c6dc54b8ull, 0x4a7a77d47f7b84b1ull, 0x48e1e9b9d588e19bull, 0x47521cc5a2e6a9e0ull,
    0x45cae0f1f545eb73ull, 0x444c0740496d4294ull, 0x42d561b3e6243d8aull, 0x4166c34c5615d0ecull,
};
static __constant__ unsigned long long kExpLo[32] = {
    0x7fffffffffffffffull, 0x7fe9d3a8e07bf086ull, 0x7fd3ab290e46d769ull, 0x7fbd867fdf0acb3bull,
    0x7fa765aca88f6453ull, 0x7f9148aec0b9b7b1ull, 0x7f7b2f857d8c51e5ull, 0x7f651a30352731eeull,
    0x7f4f08ae3dc7c426ull, 0x7f38fafeedc8dd26ull, 0x7f22f1219ba2b4aeull, 0x7f0ceb159deae091ull,
    0x7ef6e8da4b544f9aull, 0x7ee0ea6efaaf4479ull, 0x7ecaefd302e950afull, 0x7eb4f905bb0d4f78ull,
    0x7e9f06067a4360baull, 0x7e8916d497d0e3f4ull, 0x7e732b6f6b18732aull, 0x7e5d43d64b99ddd7ull,
    0x7e47600890f223deull, 0x7e31800592db7078ull, 0x7e1ba3cca92d152cull, 0x7e05cb5d2bdb84beull,
    0x7deff6b672f84e24ull, 0x7dda25d7d6b2177full, 0x7dc458c0af549908ull, 0x7dae8f7055489813ull,
    0x7d98c9e62113e1faull, 0x7d8308216b594720ull, 0x7d6d4a218cd895e5ull, 0x7d578fe5de6e95a0ull,
};
static __constant__ unsigned long long kLog[256] = {
    0x0000000000000000ull, 0x007fbfaa8ac46f01ull, 0x00fefd5358933c48ull, 0x017db6f5f8c6e761ull,
    0x01fbea8b13c03d92ull, 0x027996087816e9a6ull, 0x02f6b761284609b4ull, 0x0373d004fc3231b2ull,
    0x03efd7620b16393full, 0x046bd2e26fa28be6ull, 0x04e73ceea78842f4ull, 0x0562136c35c546e0ull,
    0x05dcda3d9ac73aadull, 0x06570a43b4333aa4ull, 0x06d0a15c48406f79ull, 0x07499d62c5890fc9ull,
    0x07c284300498a996ull, 0x083a441b14b2056bull, 0x08b2747757ae6f3full, 0x09297997c68c1f4dull,
    0x09a063cb5628b51cull, 0x0a17325f613373b9ull, 0x0a8d599f89f01e33ull, 0x0b02d754b7e1555aull,
    0x0b7835457d45a2f2ull, 0x0bece636d9c259c4ull, 0x0c6174eb21118e80ull, 0x0cd5532327ddccc6ull,
    0x0d490c9d2c4eb031ull, 0x0dbc1215f2bac54cull, 0x0e2ef047bb079d93ull, 0x0ea116eb6a028fbeull,
    0x0f1313b746795660ull, 0x0f84e5e012a79092ull, 0x0ff5fb99051e540bull, 0x1066e412d3ba6bc5ull,
    0x10d70c7d03523b42ull, 0x11470504a7c2c13eull, 0x11b6ccd551eb8f43ull, 0x122663190aeacb74ull,
    0x129532f823f522a1ull, 0x1303ce98e4c812fbull, 0x1371a0203f9f6464ull, 0x13df3ab13505f69dull,
    0x144c9d6d1a40e427ull, 0x14b9c773cae60926ull, 0x1526b7e3a9f835a8ull, 0x1592d659be06b262ull,
    0x15feb870dfd3b0a1ull, 0x166a5d42a3ad344aull, 0x16d5c3e73062139full, 0x1740eb7540ede4bdull,
    0x17ab390229d8feb1ull, 0x181544a17f67c40cull, 0x187f0d657531cff0ull, 0x18e8925ee0e73b50ull,
    0x1951d29d3c968149ull, 0x19bacd2ea90c6bc9ull, 0x1a23811ff04e5eecull, 0x1a8b4ffce877ca07ull,
    0x1af3734e9da3e5e8ull, 0x1b5b4d1e8fc9e46eull, 0x1bc23d74425dce40ull, 0x1c28e155d3498e95ull,
    0x1c8fd7c79e9a2101ull, 0x1cf5e04e25fecfcaull, 0x1d5b996b97fb5e2eull, 0x1dc1a3a0ae5d7d0full,
    0x1e26bb6e4182dcfcull, 0x1e8b80d2ebdc73baull, 0x1ef095cbde99360aull, 0x1f54b3d668b569dcull,
    0x1fb87c6dbd4ddd51ull, 0x201c930b6d7e72b9ull, 0x207fae29c9e932faull, 0x20e3163fbab04b26ull,
    0x214625c4ec31c5ccull, 0x21a8352f9b50808eull, 0x220a8ff3a4d57704ull, 0x226c8f0566523711ull,
    0x22ce31579f8be8daull, 0x232f75dc11fac43full, 0x23910482db1cf41dull, 0x23f18abcc64a04f0ull,
    0x245259f7a5d6c9c3ull, 0x24b21da226125c91ull, 0x251229280886101aull, 0x2571d175c11b0dbdull,
    0x25d1c175c24a6138ull, 0x2630a092ba0c03d7ull, 0x268f1935977e532dull, 0x26edd7c5b529954full,
    0x274c2eaafe6fbb53ull, 0x27aa1ccbc67431d7ull, 0x2808500d0e70c761ull, 0x286569d43ed44740ull,
    0x28c2c78451bd7a8full, 0x291fb9009ba39589ull, 0x297c3d2b30f51504ull, 0x29d90464c6e8d1ddull,
    0x2a34ab0ed4efeb29ull, 0x2a909387d76852e2ull, 0x2aecbe2e93b4d669ull, 0x2b47c4623bc08533ull,
    0x2ba30b7ee113780cull, 0x2bfddf6190a9bb62ull, 0x2c58f3e574d32a40ull, 0x2cb2de6654dfec97ull,
    0x2d0d083d7e692a5bull, 0x2d6771c46b3cbb12ull, 0x2dc0ad548843aa83ull, 0x2e1a274514069a80ull,
    0x2e7327edbfdfda0dull, 0x2ecc66a47ee5da65ull, 0x2f252abfbe8f444eull, 0x2f7d731484307752ull,
    0x2fd53e778123140cull, 0x302d463ba82cd4ecull, 0x30858ab43f872e41ull, 0x30dc9534b4db05d3ull,
    0x3133db0dcf147d98ull, 0x318b5c90b2d214ecull, 0x31e1a00ecd0e4041ull, 0x32381dd707140852ull,
    0x328ed6385c71ea3dull, 0x32e50b023476ec8aull, 0x333abb0260c0f902ull, 0x3390a485c1a302c0ull,
    0x33e607d98f309290ull, 0x343ae3ca0bbbdc0dull, 0x348ff82214c6e008ull, 0x34e5452cd7c3d42dull,
    0x35394735875453caull, 0x358d80852bc25747ull, 0x35e1f164b3b1c391ull, 0x3635d69da436e18cull,
    0x36892ef8291e351aull, 0x36dcbdbaef7c90f9ull, 0x3730832d2e65f4b8ull, 0x3783ba161b8b1483ull,
    0x37d6613b5b5af3f7ull, 0x38293de22be44d5aull, 0x387b894fa0fe99caull, 0x38cd42486c77d034ull,
    0x391f2f8fc533b359ull, 0x39715168cb85b7c7ull, 0x39c2df174ae8ad4aull, 0x3a14a0dcea070721ull,
    0x3a65ccfc0ad7a884ull, 0x3ab6623625d5b8dbull, 0x3b072a4b7d6e22e3ull, 0x3b58257c6b4ba197ull,
    0x3ba888099a19388full, 0x3bf850b295892688ull, 0x3c484b359070b0afull, 0x3c9877d0fe122f13ull,
    0x3ce808c3e91ee8fdull, 0x3d37cb4b377e2955ull, 0x3d86f0a49ea27a10ull, 0x3dd5778d211f40bbull,
    0x3e24febf620dd8bcull, 0x3e73167982353ef6ull, 0x3ec22ef4e2c25871ull, 0x3f0fd56e8bbdf696ull,
    0x3f5e7d1efc763ad7ull, 0x3fac82c1ef1f2328ull, 0x3ff9e510e73a0e62ull, 0x40477644cd024835ull,
    0x4095369698d3faf1ull, 0x40e251bf4070eb6full, 0x412ec67728dacadbull, 0x417c3e749abaaffeull,
    0x41c83971037c713aull, 0x421538213a383578ull, 0x42618e3d657580c8ull, 0x42ad3a7b9cf332e4ull,
    0x42f9139118e98c1eull, 0x434519b31d48fe81ull, 0x43907417c2f5bd1eull, 0x43dbfaf2c473f140ull,
    0x4427ae78b9325b4dull, 0x4472b45e26c3df47ull, 0x44bd0b56d8576c42ull, 0x45086914931d5387ull,
    0x45523b4c82e6e4ceull, 0x459d14aed11c2729ull, 0x45e73cef91aa67ebull, 0x4631903fdd7c16e1ull,
    0x467b30d1cb09a2f6ull, 0x46c4fbd6141b6e5aull, 0x470e127e6ab3e119ull, 0x475832799ef24c05ull,
    0x47a0bd7a5102b0f8ull, 0x47ea522e29be2c03ull, 0x483330465c36b02full, 0x487b56724fc51e33ull,
    0x48c4875f090d05a6ull, 0x490cffbd2928cd8dull, 0x4954be3ade3fbc1full, 0x499ca5059a0b913cull,
    0x49e4b44abcd3d27eull, 0x4a2cec37f3adfeadull, 0x4a7467fb430207faull, 0x4abc0bc0af92ab84ull,
    0x4b02f1b5939db440ull, 0x4b49ff056612bcf3ull, 0x4b9133dbf0525246ull, 0x4bd8906544f9185bull,
    0x4c1f2ccd4542f63full, 0x4c6507bf64d90243ull, 0x4cabf1e468ceb573ull, 0x4cf219e8fc0735c5ull,
    0x4d38687680ab4863ull, 0x4d7df337b25a6becull, 0x4dc3a3d5a5b7520eull, 0x4e097a79abc0061bull,
    0x4e4f774d5938669eull, 0x4e94adfa0398e416ull, 0x4eda0a2800218abcull, 0x4f1e9e801e4a2af2ull,
    0x4f6357aa411f77d3ull, 0x4fa835ce079565e8ull, 0x4fed391350b60666ull, 0x503172223ac48242ull,
    0x5075cfa14aca9cfcull, 0x50ba51b78202fc08ull, 0x50fe078c1f797ac2ull, 0x5141e145172bf614ull,
    0x5185df088a7aff8aull, 0x51c90e7d62705f15ull, 0x520c614887666b8aull, 0x524fd78f3905a02aull,
    0x52937176f1facf73ull, 0x52d63aa5e422492eull, 0x531926bfc3b856c6ull, 0x535c35e926f4d770ull,
    0x539e7247bab1b02dull, 0x53e1c77d44fde153ull, 0x5424493005c5ad2eull, 0x5465f6034919cae0ull,
    0x54a7c49a5015927bull, 0x54eaad96e69832a9ull, 0x552bc79f05b5b6f4ull, 0x556dfc52e9d02a22ull,
    0x55af59571e922ac4ull, 0x55f0d7cd24060ee9ull, 0x563277d745671facull, 0x56733e186293cbc3ull,
    0x56b42531938bdb4bull, 0x56f52d4437e96ae6ull, 0x57365671e23e74d9ull, 0x5776a35d0547c67aull,
    0x57b710a5847c97e1ull, 0x57f79e6c04ec869dull, 0x58384cd15d24397dull, 0x58781c7754b0f73cull,
};

constexpr u64 LN2_63 = 0x58b90bfbe8e7bcd6ull;  // ln 2 in units of 2^-63
constexpr double KAPPA64 = 2.885390081777926815;  // 2 log2 e

// Sum of signed terms, exact: 96 bits.
struct Acc {
  u32 w0 = 0, w1 = 0, w2 = 0;
};

#ifdef __CUDA_ARCH__
__device__ __forceinline__ void acc_add(Acc& s, u64 x, u32 ext) {  // ext: sign extension of x
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+r"(s.w0), "+r"(s.w1), "+r"(s.w2)
      : "r"((u32)x), "r"((u32)(x >> 32)), "r"(ext));
}
__device__ __forceinline__ u32 mulhi32(u32 a, u32 b) { return __umulhi(a, b); }
__device__ __forceinline__ u64 mulhi64(u64 a, u64 b) { return __umul64hi(a, b); }
__device__ __forceinline__ u64 bits_of(double d) { return (u64)__double_as_longlong(d); }
#else
inline void acc_add(Acc& s, u64 x, u32 ext) {
  unsigned __int128 v = ((unsigned __int128)s.w2 << 64) | ((u64)s.w1 << 32) | s.w0;
  v += ((unsigned __int128)ext << 64) | x;
  s.w0 = (u32)v;
  s.w1 = (u32)(v >> 32);
  s.w2 = (u32)(v >> 64);
}
inline u32 mulhi32(u32 a, u32 b) { return (u32)(((u64)a * b) >> 32); }
inline u64 mulhi64(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
inline u64 bits_of(double d) {
  union {
    double d;
    u64 u;
  } c;
  c.d = d;
  return c.u;
}
#endif

// a b / 2^64 for a, b <= 2^63, less than two units below the exact value: the
// cross products summed without the carry of the low product (their sum fits
// 64 bits because each high word is at most 2^31, and then the other operand's
// low word counts fully only if its own high word is below 2^31).
__host__ __device__ __forceinline__ u64 mul3(u64 a, u64 b) {
  const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
  const u64 t = (u64)ah * bl + (u64)al * bh;
  return (u64)ah * bh + (t >> 32);
}

constexpr int EXP_N = 1024;  // 2^{-j/1024}
constexpr int LOG_N = 256;

// Tables in shared memory (or, on the host, in plain arrays).
struct Tab {
  const u64* e;   // EXP_N entries
  const u64* l;   // LOG_N entries, -ln(R_j / 2^16)
  const u32* r;   // LOG_N entries, R_j
};

__host__ __device__ __forceinline__ u64 exp_entry(int j) {
  return mulhi64(kExpHi[j >> 5], kExpLo[j & 31]) << 1;
}
__host__ __device__ __forceinline__ u32 log_recip(int j) {
  return (u32)(((1u << 24) + 255u + j) / (256u + j));
}

#ifdef __CUDACC__
// All threads of the CTA fill the tables; a barrier has to follow.
__device__ __forceinline__ void fill_tables(u64* e, u64* l, u32* r) {
  for (int j = threadIdx.x; j < EXP_N; j += blockDim.x) e[j] = exp_entry(j);
  for (int j = threadIdx.x; j < LOG_N; j += blockDim.x) {
    l[j] = kLog[j];
    r[j] = log_recip(j);
  }
}
#endif

// 2^{-(n + F)} in units of 2^-63, F in units of 2^-63 (F < 2^63); 0 for n > 63.
__host__ __device__ __forceinline__ u64 exp2neg(u32 n, u64 F, const Tab& T) {
  constexpr u64 E1 = 3196577161300663915ull;  // l 2^72, l = ln 2 / 1024
  constexpr u64 E2 = 4431396893595737425ull;  // l^2 / 2 2^84
  constexpr u32 E3 = 3814213304u;             // l^3 / 6 2^66
  constexpr u32 E4 = 645462u;                 // l^4 / 24 2^66
  const u32 j = (u32)(F >> 53);
  const u64 x = (F << 10) & 0x7fffffffffffffffull;  // r 2^10, units of 2^-63
  const u32 x32 = (u32)(x >> 31);
  const u32 i3 = E3 - mulhi32(x32, E4);
  const u64 i2 = E2 - (((u64)x32 * i3) >> 14);
  const u64 i1 = E1 - (mul3(x, i2) >> 11);
  const u64 q = mul3(x, i1);  // units of 2^-71
  const u64 t = T.e[j];
  const u64 y = t - (mul3(t, q) >> 7);
  return n > 63u ? 0ull : y >> n;
}

// log1p(y), y <= 2^63 - 1 in units of 2^-63, as units of 2^-63.
__host__ __device__ __forceinline__ u64 log1p_fx(u64 y, const Tab& T) {
  const u32 j = (u32)(y >> 55);
  const u32 R = T.r[j];
  // t = (1 + y) R / 2^16 - 1; the terms' high bits cancel modulo 2^64
  const u64 t = (((u64)(u32)(y >> 32) * R) << 16) + (((u64)(u32)y * R) >> 16) +
                ((u64)((R << 15) - 0x80000000u) << 32);
  const u64 x = t << 7;
  const u32 x32 = (u32)(x >> 31);
  // 1/3 - x (g4 - x (g5 - x (g6 - x g7))), g_d = 2^{-7 (d - 3)} / d, units of 2^-40
  const u32 i4 = (1u << 31) - mulhi32(x32, 13421773u - mulhi32(x32, 87381u - mulhi32(x32, 585u)));
  const u64 h3 = 3074457345618258603ull - (((u64)x32 * i4) >> 9);
  const u64 h2 = (1ull << 62) - (mul3(x, h3) >> 6);
  const u64 v = mul3(mul3(x, x), h2) >> 12;  // t^2 (1/2 - t (1/3 - ..)), units of 2^-63
  return T.l[j] + t - v;
}

// The two sums of one residual over a run of samples.
struct Moments {
  Acc w, f, g;       // |w| (units of 2^-57), log1p(2^-|w|) (2^-63), w 2^(-w^2 ln2 / 8) (2^-57)
  double big = 0.0;  // |w| - 64 of samples beyond 64; not finite if a sample is not
};

__host__ __device__ __forceinline__ void moments_add(Moments& M, double w, const Tab& T) {
  const u64 b = bits_of(w);
  const u32 hi = (u32)(b >> 32);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const u32 neg = (u32)((int)hi >> 31);
  u64 W;
  if (e > 1028) {  // |w| >= 64 (|u| > 22), or not finite: the functions vanish
    M.big += __builtin_fabs(w) - 64.0;
    W = 1ull << 63;
  } else {
    const u64 m = ((b << 10) & 0x3ffffffffffffc00ull) | (e ? 1ull << 62 : 0ull);
    const int s = 1028 - e;
    W = m >> (s < 63 ? s : 63);
  }
  acc_add(M.w, W, 0u);
  acc_add(M.f, log1p_fx(exp2neg((u32)(W >> 57), (W << 6) & 0x7fffffffffffffffull, T), T), 0u);
  // w^2 ln2 / 8 from |w| in units of 2^-58, |w| < 32 (beyond, 2^-z < 2^-88)
  const u64 V = W < (1ull << 62) ? W << 1 : (1ull << 63);
  const u64 z = mul3(mul3(V, V), LN2_63);  // units of 2^-54
  u64 g = mul3(V, exp2neg((u32)(z >> 54), (z << 9) & 0x7fffffffffffffffull, T));
  g = (g ^ (((u64)neg << 32) | neg)) - ((u64)(long long)(int)neg);
  acc_add(M.g, g, neg & (g ? 0xffffffffu : 0u));
}

// a 2^64 + b as a double, signed (two's complement in hi)
__host__ __device__ __forceinline__ double to_double(u64 hi, u64 lo) {
  const bool neg = (long long)hi < 0;
  if (neg) {
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1ull : 0ull);
  }
  const double v = (double)hi * 18446744073709551616.0 + (double)lo;
  return neg ? -v : v;
}

// sum over `len` samples of log cosh u (a) and of u e^{-u^2/2} (b)
__host__ __device__ __forceinline__ void moments_sums(const Moments& M, int len, double& a,
                                                      double& b) {
  // |u| = |w| ln2 / 2: units of 2^-57, times ln2 2^63 / 2^64
  const u64 lo = ((u64)M.w.w1 << 32) | M.w.w0;
  u64 p0 = mulhi64(lo, LN2_63), p1 = 0;
  const u64 c0 = (u64)M.w.w2 * (u32)LN2_63;
  const u64 c1 = (u64)M.w.w2 * (u32)(LN2_63 >> 32) + (c0 >> 32);
  const u64 cl = (c1 << 32) | (u32)c0, ch = c1 >> 32;  // w2 LN2_63, 96 bits
  p0 += cl;
  p1 += ch + (p0 < cl ? 1ull : 0ull);
  // to units of 2^-63, plus the logarithms, minus len ln 2
  p1 = (p1 << 6) | (p0 >> 58);
  p0 <<= 6;
  const u64 f0 = ((u64)M.f.w1 << 32) | M.f.w0;
  p0 += f0;
  p1 += (u64)M.f.w2 + (p0 < f0 ? 1ull : 0ull);
  const u64 n0 = (u64)(u32)len * (u32)LN2_63;
  const u64 n1 = (u64)(u32)len * (u32)(LN2_63 >> 32) + (n0 >> 32);
  const u64 nl = (n1 << 32) | (u32)n0, nh = n1 >> 32;
  p1 -= nh + (p0 < nl ? 1ull : 0ull);
  p0 -= nl;
  a = to_double(p1, p0) * 0x1p-63 + M.big * (1.0 / KAPPA64);
  const u64 g0 = ((u64)M.g.w1 << 32) | M.g.w0;
  // big is zero unless samples lie beyond 64; not finite makes b NaN
  b = to_double((u64)(long long)(int)M.g.w2, g0) * (0x1p-57 / KAPPA64) + M.big * 0.0;
}

}  // namespace fx
}  // namespace vl
