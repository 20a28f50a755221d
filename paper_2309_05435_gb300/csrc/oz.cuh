// Binary64 products on the bf16 tensor cores by digit products (the
// splitting of Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012).
//
// A row of an operand with exponent E (|x_k| 2^s_k < 2^E for all its entries) is
// held as 62-bit integers X_k = rint(x_k 2^(62 + s_k - E)), and X as eight signed
// base-256 digits, X = sum_i d_i 256^(7 - i) with |d_0| <= 65 and -128 <= d_i <= 127:
// exact bf16 values.  The tensor cores sum d_i e_j products in FP32; over K <=
// kChunk the sums of the products with the same i + j = s stay below 2^24 in
// magnitude, so they are exact integers, and
//   x . y = 2^(Ea + Eb - 12) sum_s 256^-s g_s,  g_s = sum_{i + j = s} d_i . e_j.
// Products with i + j > 7 (below 2^-60 of the largest one) are dropped.  What
// remains is the 62-bit rounding of the operands and one rounding to binary64
// at the end: for entries within 2^-8 of their row's largest that is below the
// error of a binary64 FMA chain.
//
// The shifts s_k are what keeps the entries of a row within that range whatever
// the units of the unknowns: the two operands of a product carry them with
// opposite signs, so that they cancel in it.  They are read off a symmetric
// positive definite matrix M over the contracted index (half_exponent of M_kk): a
// row of M satisfies |M_ik| <= sqrt(M_ii M_kk), so its entries with s_k = -log2
// sqrt(M_kk) all lie below sqrt(M_ii), and the other operand's entries, which
// scale like 1 / sqrt(M_kk), are as even.  A rescaling x -> D x of the unknowns by
// powers of two therefore changes no digit, and no bit of a result but its
// exponent.  Without the shifts D Q D lost what the spread of D exceeded 2^8 by
// (emulated, diagonal of a 192 x 192 inverse: 4e-12 relative for D over 10^-4 .. 10^4,
// 1e-7 over 10^-6 .. 10^6, 7e-5 over 10^-8 .. 10^8; 1e-15 with them).
#pragma once

#include <cstdint>

namespace qsel {
namespace oz {

constexpr int kDigits = 8;
constexpr int kChunk = 128;                   // K of an exact FP32 sum: 7 kChunk 2^14 < 2^24
constexpr int32_t kNonFinite = 0x7fffffff;    // exponent of a row with an infinity or a NaN

// Largest exponent field of x_u 2^(SIGN sh_u) (fields lie in 0 .. 0x7ff, shifts
// within +- 2048), kBadField where an infinity or a NaN is among them; a row's
// largest decides its exponent, from kNoField on.  Zeros count as 2^-1023: with
// shifts of M's diagonal the entries that matter lie far above it.
constexpr int kNoField = -(1 << 16), kBadField = 1 << 16;
template <int SIGN, int N>
__device__ __forceinline__ int max_field(const double (&x)[N], const int (&sh)[N]) {
  int hi = 0, s = kNoField;
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const int f = (__double2hiint(x[u]) >> 20) & 0x7ff;
    hi = max(hi, f);
    s = max(s, f + SIGN * sh[u]);
  }
  return hi == 0x7ff ? kBadField : s;
}
// The row exponent E of a largest scaled field (see above).
__device__ __forceinline__ int32_t row_exponent(int field) { return field == kBadField ? kNonFinite : field - 1022; }
// The exponent that the digits of a row are formed with: all zero in a row with an
// infinity or a NaN.
__device__ __forceinline__ int32_t digit_exponent(int32_t E) { return E == kNonFinite ? 1 << 16 : E; }

// log2(sqrt(v)) to the nearest integer or the next one, for a positive normal v, else 0.
__device__ __forceinline__ int half_exponent(double v) {
  const int f = __double2hiint(v) >> 20;   // with the sign
  return f > 0 && f < 0x7ff ? (f >> 1) - 511 : 0;
}
// floor(log2 |v|) for a normal v, else 0.
__device__ __forceinline__ int full_exponent(double v) {
  const int f = (__double2hiint(v) >> 20) & 0x7ff;
  return f > 0 && f < 0x7ff ? f - 1023 : 0;
}

// rint(x 2^(62 - E)) for |x| < 2^E (ties away from zero), in integer arithmetic:
// GB300 runs binary64 at 1/64 of the integer rate.  E is the row's digit exponent
// less the entry's shift.
__device__ __forceinline__ int64_t fixed62(double x, int32_t E) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
  const int field = (int)(bits >> 52) & 0x7ff;
  // |x| = m 2^(field - 1075), also for field 0
  const uint64_t frac = bits & 0x000fffffffffffffULL;
  const uint64_t m = field ? frac | 0x0010000000000000ULL : frac << 1;
  // m 2^10 shifted right by one more than the distance to the largest exponent;
  // out of range (below zero only for x = 0 or in an empty row) gives 0
  const uint32_t d = (uint32_t)(E + 1022 - field), r = min(d, 62u);
  const uint64_t v = d > 62u ? 0 : ((m << 10) + (1ULL << r)) >> (r + 1);
  return (bits >> 63) ? -(int64_t)v : (int64_t)v;
}

// The bytes of a fixed62 value from which digit_f forms the digits: one 64-bit
// addition carries every digit's sign (each byte is its digit + 128).
__device__ __forceinline__ uint2 digit_bytes(int64_t X) {
  const uint64_t y = ((uint64_t)X + 0x0080808080808080ULL) ^ 0x8000000000000000ULL;
  return make_uint2((uint32_t)y, (uint32_t)(y >> 32));
}
// Digit i as a float: byte 7 - i of y placed in the low mantissa byte of 2^23.
template <int I>
__device__ __forceinline__ float digit_f(uint2 y) {
  constexpr uint32_t byte = (7 - I) & 3;
  const uint32_t w = I < 4 ? y.y : y.x;
  return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u + byte)) - 8388736.0f;
}
// Digit I of two neighbouring values as packed bf16 (first value in the low half).
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint2 a, uint2 b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(digit_f<I>(b)), "f"(digit_f<I>(a)));
  return r;
}

// The digit sums of one output element: sum_s 256^-s g_s = (hi + lo 2^-32) 2^-24,
// both exact over K up to 16384.
__device__ __forceinline__ void acc_hi(int64_t &hi, int g0, int g1, int g2, int g3) {
  hi += (int64_t)(g0 * 256 + g1) * 65536 + (g2 * 256 + g3);
}
__device__ __forceinline__ void acc_lo(int64_t &lo, int g4, int g5, int g6, int g7) {
  lo += ((int64_t)g4 * 16777216 + (int64_t)g5 * 65536) + ((int64_t)g6 * 256 + g7);
}

// +- (hi + lo 2^-32) 2^(Ea + Eb - 36) rounded once to binary64 (to nearest, ties
// to even), in integer arithmetic: hi 2^32 + lo as a 96-bit magnitude H 2^32 + L,
// normalised to 64 bits.  Two conversions, an FMA and a scaling in binary64
// would take 4 of the 2 binary64 operations per cycle that the SM has for all
// its threads; this takes about 40 integer operations at 64 or more per cycle.
__device__ __forceinline__ double value(int64_t hi, int64_t lo, int32_t Ea, int32_t Eb, bool negate) {
  const int64_t h = hi + (lo >> 32);
  const uint32_t l = (uint32_t)lo;
  const bool neg = h < 0;
  uint64_t H = neg ? ~(uint64_t)h + (l == 0 ? 1 : 0) : (uint64_t)h;
  uint64_t L = (uint64_t)(neg ? 0u - l : l) << 32;
  int x = Ea + Eb - 25;                       // exponent of bit 11 of the top word before normalising
  if (H == 0) {
    H = L;
    L = 0;
    x -= 64;
  }
  if (Ea == kNonFinite || Eb == kNonFinite) return __longlong_as_double(0x7ff8000000000000LL);
  if (H == 0) return 0.0;
  const int z = __clzll((long long)H);
  const uint64_t T = z ? (H << z) | (L >> (64 - z)) : H;
  const bool rest = (L << z) != 0;
  uint64_t keep = T >> 11;
  const uint32_t rem = (uint32_t)T & 0x7ffu;
  keep += (rem > 0x400u || (rem == 0x400u && (rest || (keep & 1)))) ? 1 : 0;
  x -= z;
  const int e = x + 1074;                     // the exponent field less one; keep carries the one
  const uint64_t sign = (neg != negate) ? 0x8000000000000000ULL : 0;
  if (e >= 0 && e < 2045) return __longlong_as_double((long long)((((uint64_t)e) << 52) + keep) | (long long)sign);
  const double v = ldexp((double)keep, x);    // overflows to infinity, or rounds to a subnormal
  return sign ? -v : v;
}

// kind::f16 with bf16 operands and FP32 accumulation, M = 128, both operands
// K-major: D format F32 (bit 4), A and B bf16 (bits 7, 10), N >> 3 at bit 17,
// M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(id), "r"(accumulate)
      : "memory");
}
// K-major operand with rows of `row_bytes` (64 or 128) and the swizzle of that
// width; 8-row groups 8 row_bytes apart, descriptor version 1.
template <int ROW_BYTES>
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  static_assert(ROW_BYTES == 64 || ROW_BYTES == 128, "swizzle width");
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)((8 * ROW_BYTES) >> 4) << 32;     // stride byte offset
  d |= (uint64_t)1 << 46;                          // descriptor version
  d |= (uint64_t)(ROW_BYTES == 128 ? 2 : 4) << 61; // SWIZZLE_128B / SWIZZLE_64B
  return d;
}

// The digit products of one K = 16 step: A holds digits i as consecutive 128-row
// tiles (a_tile bytes each), B digits j as consecutive 64-row tiles (b_tile
// bytes each).  Digit i times the stacked digits j .. of B lands in the column
// groups i + j of the accumulator: one MMA of up to 256 columns serves up to
// four digit pairs, and A is read 12 times instead of 36.
template <int ROW_BYTES>
__device__ __forceinline__ void mma_digits(uint32_t d, uint32_t a, uint32_t b, uint32_t a_tile, uint32_t b_tile,
                                           bool first) {
#pragma unroll
  for (int i = 0; i < kDigits; ++i) {
#pragma unroll
    for (int j = 0; j < kDigits - i; j += 4) {
      const int cnt = (kDigits - i - j) < 4 ? (kDigits - i - j) : 4;
      mma_bf16(d + 64u * (i + j), smem_desc<ROW_BYTES>(a + i * a_tile), smem_desc<ROW_BYTES>(b + j * b_tile),
               idesc(64 * cnt), (first && i == 0) ? 0u : 1u);
    }
  }
}

// Columns t0 .. + 7 of four accumulator groups (64 columns apart) as integers.
// The loads and their wait are one statement, so that no use of a value moves
// between them.
__device__ __forceinline__ void load_groups(uint32_t t0, int (&g)[4][8]) {
  uint32_t v[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%33];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16, %17, %18, %19, %20, %21, %22, %23}, [%34];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24, %25, %26, %27, %28, %29, %30, %31}, [%35];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(t0), "r"(t0 + 64u), "r"(t0 + 128u), "r"(t0 + 192u)
      : "memory");
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < 8; ++c) g[q][c] = __float2int_rn(__uint_as_float(v[8 * q + c]));
}

// Adds the accumulator columns t .. + 7 (all eight groups) to hi, lo.
__device__ __forceinline__ void accumulate8(uint32_t t, int64_t *hi, int64_t *lo) {
  int g[4][8];
  load_groups(t, g);
#pragma unroll
  for (int c = 0; c < 8; ++c) acc_hi(hi[c], g[0][c], g[1][c], g[2][c], g[3][c]);
  load_groups(t + 256u, g);
#pragma unroll
  for (int c = 0; c < 8; ++c) acc_lo(lo[c], g[0][c], g[1][c], g[2][c], g[3][c]);
}

}  // namespace oz
}  // namespace qsel
