// The analysis's Ozaki form: float64 results from exact products of bf16 digits,
// and the sums of its levels (k_oz_analysis).  Included by yy_tc_pair.cuh after the
// PTX wrappers it uses.
#pragma once

namespace yy {

// Float64 results by the Ozaki scheme: each operand row is scaled by a power
// of two to |x| <= 1/2 and written with six balanced base-256 digits,
// x = sum_s a_s 2^(-8 (s + 1)) + r, integers |a_s| <= 128 (the first up to 256 for the sums
// of two cells; exact in bf16), |r| <= 2^-49: the digits of round(x 2^48), each in
// [-127, 128] with a carry into the next.  The products of digit levels
// L = s + t <= 6 (26 of the 36) are kept; the dropped ones add up to below 2^-56.  A
// level has at most 6 products, one with a first digit of the cells, so over K <= 146
// columns it stays below 7 * 146 * 2^14 < 2^24 and accumulates exactly in fp32.
// Longer K runs in several fills, which the epilogue adds.  The epilogue combines
// levels 0-3 in int64 and the three lowest in fp32, and rounds once to float64.  The
// digits are rounded to nearest, so their representation errors take either
// sign and grow like sqrt(K) along K rather than like K.
struct FormOzaki {
  typedef __nv_bfloat16 elem;
  static constexpr int kKind = KIND_BF16, kElem = 2, kPA = 6, kPB = 6, kAccs = 7;
  static constexpr int kMaxK = 640;   // cells of the longest row taken: up to three fills a class
};

// v 2^e exactly, for |v| < 2^53 and a result in the normal range, built
// from the bits: |v| shifted so that its top bit lands on bit 52 (the
// implicit one), then the biased exponent less one added above it (the
// implicit one carries it up by one) and the sign bit set; anything else
// takes ldexp.
__device__ __forceinline__ double i64_ldexp(long long v, int e) {
  const unsigned long long s = (unsigned long long)(v >> 63);          // 0 or all ones
  const unsigned long long u = ((unsigned long long)v ^ s) - s;        // |v|
  const int lz = __clzll((long long)u);                                // 64 for v = 0
  const int be = 1086 - lz + e;                                        // (63 - lz) + 1023 + e
  if (lz < 11 || lz == 64 || be <= 0 || be >= 2047) return lz == 64 ? 0.0 : ldexp((double)v, e);
  const unsigned long long m = u << (lz - 11);
  return __longlong_as_double((long long)((m + ((unsigned long long)(be - 1) << 52)) | (s << 63)));
}

// i64_ldexp for callers that checked e once per row: |v| < 2^53 and
// e in [-1022, 971] keep every nonzero result normal, so the range checks go.
__device__ __forceinline__ bool i64_ldexp_row_ok(int e) { return e >= -1022 && e <= 971; }
__device__ __forceinline__ double i64_ldexp_row(long long v, int e) {
  const unsigned long long s = (unsigned long long)(v >> 63);
  const unsigned long long u = ((unsigned long long)v ^ s) - s;
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << ((lz - 11) & 63);
  const unsigned long long b = (m + ((unsigned long long)(1085 - lz + e) << 52)) | (s << 63);
  return __longlong_as_double((long long)(u == 0ull ? 0ull : b));
}

// i64_ldexp_row for |v| < 2^54, rounded to nearest even (e in [-1022, 970]): the
// top bit on bit 53, so that the bit below the last one decides.
__device__ __forceinline__ double i64_ldexp_row54(long long v, int e) {
  const unsigned long long s = (unsigned long long)(v >> 63);
  const unsigned long long u = ((unsigned long long)v ^ s) - s;
  const int lz = __clzll((long long)u);
  const unsigned long long t = u << ((lz - 10) & 63);
  const unsigned long long m = (t + ((t >> 1) & 1)) >> 1;   // a carry into bit 53 steps the exponent
  const unsigned long long b = (m + ((unsigned long long)(1085 - lz + e) << 52)) | (s << 63);
  return __longlong_as_double((long long)(u == 0ull ? 0ull : b));
}

// The same through the float64 pipe's conversion (to nearest; exact for |v| < 2^53) and an
// exponent add: a few issue slots instead of the integer formatting, for
// callers that spread their values over both pipes.
__device__ __forceinline__ double i64_ldexp_row_cvt(long long v, int e) {
  const double d = __ll2double_rn(v);
  const int hi = __double2hiint(d);   // zero for v = 0 alone
  return __hiloint2double(hi == 0 ? 0 : hi + (int)((unsigned)e << 20), __double2loint(d));
}

// An accumulator value of the Ozaki forms: an integer below 2^24 held in fp32.
__device__ __forceinline__ int oz_int(uint32_t v) { return __float2int_rn(__uint_as_float(v)); }

// Level sum S_L of 8 columns (accumulator L, bn columns apart from tcol
// onwards), as an integer and as the fp32 value itself.
__device__ __forceinline__ void oz_level(uint32_t tcol, int bn, int L, int (&S)[8]) {
  uint32_t v[8];
  tmem_ld8_async(tcol + (uint32_t)(L * bn), v);
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < 8; ++j) S[j] = oz_int(v[j]);
}

__device__ __forceinline__ void oz_level_f(uint32_t tcol, int bn, int L, float (&S)[8]) {
  uint32_t v[8];
  tmem_ld8_async(tcol + (uint32_t)(L * bn), v);
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < 8; ++j) S[j] = __uint_as_float(v[j]);
}

// exact float64 of an fp32 value times 2^e (a normal result; zero stays zero)
__device__ __forceinline__ double f32_ldexp(float f, int e) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t ex = (u >> 23) & 0xFFu;
  if (ex == 0u) return 0.0;   // the values here are integer combinations: zero or at least 1
  const int be = (int)ex + 896 + e;
  if (ex == 255u || be <= 0 || be >= 2047) return ldexp((double)f, e);
  const unsigned long long bits = ((unsigned long long)(u & 0x80000000u) << 32) | ((unsigned long long)be << 52) |
                                  ((unsigned long long)(u & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)bits);
}

// One fill's level sums S_0 .. S_6 of 8 columns (TMEM column tcol) added to
// the chunk's running value 2^ce (hi 2^24 + lo):
//   hi += S_0 2^24 + S_1 2^16 + S_2 2^8 + S_3   (int64: below 2^48 per fill)
//   lo += S_4 2^16 + S_5 2^8 + S_6             (fp32)
// hi stays exact (below 2^50 over four fills, exact in float64 too).  lo is
// formed in fp32 from the accumulator values (a unit is 2^-64 of the two
// rows' scales): below 2^40 units per fill, so its rounding stays under 2^18
// units over four fills, below the digits' own error, which is up to 2^15
// units per product term (2^-49 of the scales) and adds up over the K terms.
__device__ __forceinline__ void ozaki_accumulate(uint32_t tcol, int bn, long long (&hi)[8], float (&lo)[8]) {
  int S[8];
  oz_level(tcol, bn, 0, S);
#pragma unroll
  for (int j = 0; j < 8; ++j) hi[j] += (long long)S[j] << 24;
  oz_level(tcol, bn, 1, S);
#pragma unroll
  for (int j = 0; j < 8; ++j) hi[j] += (long long)S[j] << 16;
  oz_level(tcol, bn, 2, S);
#pragma unroll
  for (int j = 0; j < 8; ++j) hi[j] += (long long)S[j] << 8;
  oz_level(tcol, bn, 3, S);
#pragma unroll
  for (int j = 0; j < 8; ++j) hi[j] += (long long)S[j];
  float u[8], w[8];
  oz_level_f(tcol, bn, 4, u);
  oz_level_f(tcol, bn, 5, w);
#pragma unroll
  for (int j = 0; j < 8; ++j) u[j] = fmaf(w[j], 256.0f, u[j] * 65536.0f);
  oz_level_f(tcol, bn, 6, w);
#pragma unroll
  for (int j = 0; j < 8; ++j) lo[j] += u[j] + w[j];
}

// The chunk's float64 values: one rounding, in the final addition.
__device__ __forceinline__ void ozaki_finish(const long long (&hi)[8], const float (&lo)[8], int ce, double *dst) {
#pragma unroll
  for (int j = 0; j < 8; ++j) dst[j] = i64_ldexp(hi[j], ce + 24) + f32_ldexp(lo[j], ce);
}

}  // namespace yy
