// Residue arithmetic of the emulated FP64 products (Ozaki scheme II: K. Ozaki,
// Y. Uchino, T. Imamura, "Ozaki Scheme II: A GEMM-oriented emulation of
// floating-point matrix multiplication using an integer modular technique",
// 2025; the arithmetic below is written from the Chinese remainder theorem).
//
// Both operands are integers of at most 2^kOzFrac (fixed point relative to a
// row's and a column's largest entry).  Their product is an integer S with
// |S| <= K 2^(2 kOzFrac), recovered from its residues modulo kOzP pairwise
// coprime moduli p_l whose product P exceeds 2 |S|: one tensor-core product of
// residues per modulus, where cutting the same integers into digits takes one
// per digit pair (17 against 55 products of the same K).
//
// Residues are balanced (|r| <= 128), exact in BF16, and a product of two is at
// most 2^14, so FP32 sums of kOzChunk = 2^10 of them are exact integers below
// or at 2^24.  The left operand's residues carry the factor (P / p_l)^-1 mod
// p_l, so that with c_l = (sum mod p_l)
//     S = sum_l c_l P / p_l  (mod P).
// The moduli are grouped by three (group products Q_g < 2^24): 32-bit integer
// sums n_g inside a group, then S / P = sum_g n_g / Q_g (mod 1) in 128-bit fixed
// point, whose wrap-around takes off the multiple of P by itself (|S| / P stays
// below 1/3).  Its error, 2^28 units of 2^-128, is 2^33 in S, far below the
// 2^59 that rounding one operand entry costs; |S| below 2^37 counts as zero, so
// that an exact zero stays one.
#pragma once

#include <stdint.h>

namespace {

constexpr int kOzP = 17;            // moduli
constexpr int kOzFrac = 59;         // fraction bits of the fixed-point operands
constexpr int kOzChunk = 1024;      // K per exact FP32 sum
constexpr int kOzMaxK = 8192;       // K per product: K 2^(2 kOzFrac) < P / 3
constexpr int kOzGroups = 6;        // groups of three moduli (the last: two)
// residue bytes of a 128 x 256 tile in words, per modulus and in all; a CTA's
// scratch holds two tiles (one being written, one being converted)
constexpr int kOzPlaneWords = (256 / 4) * 128;
constexpr int kOzTileWords = kOzP * kOzPlaneWords;
__device__ __forceinline__ size_t oz_scratch_at(int cta, int half, int col) {
  return (size_t)(2 * cta + half) * kOzTileWords + (size_t)(col / 4) * 128;
}

// Operands with infinities or NaNs: a row of the left operand that holds one has
// the exponent kOzExpBad; a column of the right one whose first one is at k has
// (k + 1) << 16 added to the low half of its exponent.  Either takes an entry's
// exponent past kOzExpFlag (finite operands stay below 2^13), and the conversion
// writes NaN: to the whole row, and to the column from row k on (a triangular
// product does not multiply it above) or, of a full product, to all of it.
constexpr int kOzExpBad = 1 << 20, kOzExpFlag = 1 << 14;
__host__ __device__ constexpr int oz_flag_column(int e, int k) { return ((k + 1) << 16) | (e & 0xffff); }

struct OzTables {
  // slicing: balanced weights (2^15)^j of the four 15-bit limbs, for the left
  // operand times (P / p_l)^-1, modulo p_l
  float wa[kOzP][4], wx[kOzP][4];
  float modf[kOzP], inv[kOzP];
  uint32_t gw[kOzP];             // Q_g / p_l
  uint32_t F[kOzGroups][4];      // 2^128 / Q_g
  uint32_t init[4];              // -sum_l 128 2^128 / p_l: undoes the offset of the stored bytes
};

constexpr uint32_t kOzMod[kOzP] = {256, 251, 249, 247, 245, 241, 239, 233, 229, 227, 223, 211, 199, 197, 193, 191, 187};

struct U160 {
  uint32_t w[5];
};

constexpr U160 u160_mul(U160 a, uint32_t m) {
  U160 r{};
  uint64_t c = 0;
  for (int i = 0; i < 5; ++i) {
    c += (uint64_t)a.w[i] * m;
    r.w[i] = (uint32_t)c;
    c >>= 32;
  }
  return r;
}

constexpr U160 u160_add(U160 a, U160 b) {
  U160 r{};
  uint64_t c = 0;
  for (int i = 0; i < 5; ++i) {
    c += (uint64_t)a.w[i] + b.w[i];
    r.w[i] = (uint32_t)c;
    c >>= 32;
  }
  return r;
}

// round(2^128 num / den) for num < den < 2^26, four words
constexpr U160 u128_fraction(uint32_t num, uint32_t den) {
  U160 r{};
  uint64_t rem = num;
  for (int i = 3; i >= 0; --i) {
    rem <<= 32;
    r.w[i] = (uint32_t)(rem / den);
    rem %= den;
  }
  U160 one{{2 * rem >= den ? 1u : 0u, 0, 0, 0, 0}};
  return u160_add(r, one);
}

// representative of v modulo p in (-p/2, p/2]
constexpr int oz_balance(uint32_t v, uint32_t p) { return 2 * v > p ? (int)v - (int)p : (int)v; }

constexpr OzTables oz_make_tables() {
  OzTables t{};
  U160 off{};
  for (int l = 0; l < kOzP; ++l) {
    const uint32_t p = kOzMod[l];
    uint32_t rest = 1;  // P / p_l mod p_l
    for (int k = 0; k < kOzP; ++k)
      if (k != l) rest = rest * (kOzMod[k] % p) % p;
    uint32_t inv = 1;
    while (rest * inv % p != 1) ++inv;  // coprime moduli: ends below p
    uint32_t x = 1;
    for (int j = 0; j < 4; ++j) {
      t.wx[l][j] = (float)oz_balance(x, p);
      t.wa[l][j] = (float)oz_balance(x * inv % p, p);
      x = x * (32768 % p) % p;
    }
    t.modf[l] = (float)p;
    t.inv[l] = 1.0f / (float)p;
    off = u160_add(off, u128_fraction(128 % p, p));
  }
  for (int g = 0; g < kOzGroups; ++g) {
    uint32_t Q = 1;
    for (int l = 0; l < kOzP; ++l)
      if (l / 3 == g) Q *= kOzMod[l];
    for (int l = 0; l < kOzP; ++l)
      if (l / 3 == g) t.gw[l] = Q / kOzMod[l];
    const U160 f = u128_fraction(1, Q);
    for (int i = 0; i < 4; ++i) t.F[g][i] = f.w[i];
  }
  uint64_t c = 1;
  for (int i = 0; i < 4; ++i) {
    c += (uint32_t)~off.w[i];
    t.init[i] = (uint32_t)c;
    c >>= 32;
  }
  return t;
}

constexpr OzTables kOzTables = oz_make_tables();
__constant__ OzTables c_oz = kOzTables;

constexpr U160 oz_product_of_moduli() {
  U160 P{{1, 0, 0, 0, 0}};
  for (int l = 0; l < kOzP; ++l) P = u160_mul(P, kOzMod[l]);
  return P;
}

constexpr bool oz_moduli_ok() {
  for (int a = 0; a < kOzP; ++a)
    for (int b = a + 1; b < kOzP; ++b) {
      uint32_t x = kOzMod[a], y = kOzMod[b];
      while (y != 0) {
        const uint32_t z = x % y;
        x = y;
        y = z;
      }
      if (x != 1) return false;
    }
  // 3 kOzMaxK 2^(2 kOzFrac) = 3 * 2^131 <= P, and 2^132 <= P < 2^133
  const U160 P = oz_product_of_moduli();
  return P.w[4] >= 3u * (kOzMaxK >> 10) && P.w[4] >= 16u && P.w[4] < 32u;
}
static_assert(2 * kOzFrac + 10 == 128 && oz_moduli_ok(), "coprime moduli whose product covers the largest sum");

// the leading 64 bits of P (2^132 <= P < 2^133)
constexpr uint64_t oz_lead_p() {
  const U160 P = oz_product_of_moduli();
  return (uint64_t)P.w[4] << 59 | (uint64_t)P.w[3] << 27 | P.w[2] >> 5;
}
constexpr uint64_t kOzLeadP = oz_lead_p();

// Balanced residue of an exact integer v, |v| <= 2^24: the quotient is rounded
// with one FP32 rounding each for v / p and the sum with 1.5 2^23, so the result
// may pass p / 2 by 1% of p; |r| <= 128 (r = 128 only for p = 256, where the
// stored byte wraps to the congruent -128).
__device__ __forceinline__ float oz_residue(float v, float mod, float inv) {
  const float q = __fadd_rn(fmaf(v, inv, 12582912.0f), -12582912.0f);
  return fmaf(-mod, q, v);
}

// four small integers as signed bytes
__device__ __forceinline__ uint32_t oz_pack_bytes(const float (&r)[4]) {
  uint32_t b[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) b[j] = __float_as_uint(__fadd_rn(r[j], 12582912.0f));
  return __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
}

// r += the signed bytes of w, reduced again
__device__ __forceinline__ void oz_add_bytes(float (&r)[4], uint32_t w, float mod, float inv) {
  const uint32_t u = w ^ 0x80808080u;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float old = __fadd_rn(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440 | j)), -8388736.0f);
    r[j] = oz_residue(__fadd_rn(r[j], old), mod, inv);
  }
}

// The integer S whose residues c_l + 128 are byte j of w[l]: the 64 leading bits
// of S / P times those of P (relative error below 2^-61), rounded once to 53
// bits.  Returned as a double in [1, 2) (or 2 after rounding up; 0 for S = 0)
// with S's sign and the exponent of its leading bit in e.  Written without
// branches so that the conversions of several results overlap.
__device__ __forceinline__ uint64_t oz_crt(const uint32_t (&w)[kOzP], int j, int &e) {
  uint64_t acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = c_oz.init[i];
#pragma unroll
  for (int g = 0; g < kOzGroups; ++g) {
    uint32_t ng = 0;
#pragma unroll
    for (int l = 3 * g; l < 3 * g + 3 && l < kOzP; ++l) ng += __byte_perm(w[l], 0u, 0x4440 | j) * c_oz.gw[l];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] += (uint64_t)ng * c_oz.F[g][i];
  }
  acc[1] += acc[0] >> 32;
  acc[2] += acc[1] >> 32;
  acc[3] += acc[2] >> 32;
  uint64_t lo = acc[1] << 32 | (uint32_t)acc[0], hi = acc[3] << 32 | (uint32_t)acc[2];
  // magnitude (of a negative value less one unit of 2^-128, far below the error)
  const uint32_t sign = (uint32_t)(hi >> 63);
  const uint64_t flip = sign ? ~0ull : 0ull;
  hi ^= flip;
  lo ^= flip;
  const bool small = hi == 0;
  const bool zero = small && (lo >> 32) == 0;
  hi = small ? lo : hi;
  lo = small ? 0ull : lo;
  const int z = __clzll((long long)hi);
  const uint64_t m = hi << (z & 63) | (lo >> 1) >> (63 - (z & 63));
  uint64_t h = __umul64hi(m, kOzLeadP);  // in [2^62, 2^64)
  const uint32_t up = (uint32_t)(h >> 63);
  e = 131 + (int)up - z - (small ? 64 : 0);
  h <<= 1 - up;
  const uint64_t r = (h >> 11) + ((h >> 10) & 1);
  // r's bit 52 (or 53) carries into the exponent field
  return zero ? 0ull : (((uint64_t)(sign << 11) + 1022) << 52) + r;
}

// y 2^e for y from oz_crt (ldexp's rounding below the normal range)
__device__ __forceinline__ bool oz_scales(int e) { return e >= -1022 && e <= 1022; }
__device__ __forceinline__ double oz_scaled(uint64_t y, int e) {
  return __longlong_as_double((long long)(y == 0 ? 0ull : y + ((uint64_t)(int64_t)e << 52)));
}

}  // namespace
