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
// sums inside a group, six multiword terms n_g P / Q_g, and a multiple of P
// found in FP32 from sum_g n_g / Q_g (|S| / P stays below 1/3, so rounding to
// the nearest integer has a margin of 1/6).
#pragma once

#include <stdint.h>

namespace {

constexpr int kOzP = 17;            // moduli
constexpr int kOzFrac = 59;         // fraction bits of the fixed-point operands
constexpr int kOzChunk = 1024;      // K per exact FP32 sum
constexpr int kOzMaxK = 8192;       // K per product: K 2^(2 kOzFrac) < P / 3
constexpr int kOzGroups = 6;        // groups of three moduli (the last: two)
constexpr int kOzTileWords = kOzP * (256 / 4) * 128;  // residue bytes of a 128 x 256 tile, in words

struct OzTables {
  // slicing: balanced weights (2^15)^j of the four 15-bit limbs, for the left
  // operand times (P / p_l)^-1, modulo p_l
  float wa[kOzP][4], wx[kOzP][4];
  float modf[kOzP], inv[kOzP];
  uint32_t gw[kOzP];             // Q_g / p_l
  uint32_t W[kOzGroups][4];      // P / Q_g (below 2^128)
  float qinv[kOzGroups];         // 1 / Q_g
  uint32_t negP[5];              // 2^160 - P
  uint32_t init[5];              // 16 P - sum_l 128 P / p_l (mod 2^160): undoes the offset of the
                                 // stored bytes; 16 P keeps the multiple of P taken off positive
  float init_f;                  // 16 - sum_l 128 / p_l
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

constexpr U160 u160_neg(U160 a) {
  U160 r{};
  uint64_t c = 1;
  for (int i = 0; i < 5; ++i) {
    c += (uint32_t)~a.w[i];
    r.w[i] = (uint32_t)c;
    c >>= 32;
  }
  return r;
}

// representative of v modulo p in (-p/2, p/2]
constexpr int oz_balance(uint32_t v, uint32_t p) { return 2 * v > p ? (int)v - (int)p : (int)v; }

constexpr OzTables oz_make_tables() {
  OzTables t{};
  U160 P{{1, 0, 0, 0, 0}};
  for (int l = 0; l < kOzP; ++l) P = u160_mul(P, kOzMod[l]);
  U160 off{};
  float off_f = 0.0f;
  for (int l = 0; l < kOzP; ++l) {
    const uint32_t p = kOzMod[l];
    U160 part{{1, 0, 0, 0, 0}};
    uint32_t rest = 1;
    for (int k = 0; k < kOzP; ++k)
      if (k != l) {
        part = u160_mul(part, kOzMod[k]);
        rest = rest * (kOzMod[k] % p) % p;
      }
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
    off = u160_add(off, u160_mul(part, 128));
    off_f -= 128.0f / (float)p;
  }
  for (int g = 0; g < kOzGroups; ++g) {
    uint32_t Q = 1;
    U160 W{{1, 0, 0, 0, 0}};
    for (int l = 0; l < kOzP; ++l) {
      if (l / 3 == g)
        Q *= kOzMod[l];
      else
        W = u160_mul(W, kOzMod[l]);
    }
    for (int l = 0; l < kOzP; ++l)
      if (l / 3 == g) t.gw[l] = Q / kOzMod[l];
    for (int i = 0; i < 4; ++i) t.W[g][i] = W.w[i];
    t.qinv[g] = 1.0f / (float)Q;
  }
  const U160 nP = u160_neg(P), io = u160_add(u160_neg(off), u160_mul(P, 16));
  for (int i = 0; i < 5; ++i) {
    t.negP[i] = nP.w[i];
    t.init[i] = io.w[i];
  }
  t.init_f = off_f + 16.0f;
  return t;
}

constexpr OzTables kOzTables = oz_make_tables();
__constant__ OzTables c_oz = kOzTables;

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
  U160 P{{1, 0, 0, 0, 0}};
  for (int l = 0; l < kOzP; ++l) P = u160_mul(P, kOzMod[l]);
  // 3 kOzMaxK 2^(2 kOzFrac) = 3 * 2^131 <= P < 2^133 (so every P / Q_g fits four words)
  return P.w[4] >= 3u * (kOzMaxK >> 10) && P.w[4] < 32u;
}
static_assert(2 * kOzFrac + 10 == 128 && oz_moduli_ok(), "coprime moduli whose product covers the largest sum");

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

// The integer whose residues c_l + 128 are byte j of w[l], times 2^shift, as a
// correctly rounded double (ldexp's rounding below the normal range).
__device__ __forceinline__ double oz_crt(const uint32_t (&w)[kOzP], int j, int shift) {
  uint64_t acc[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) acc[i] = c_oz.init[i];
  float f = c_oz.init_f;
#pragma unroll
  for (int g = 0; g < kOzGroups; ++g) {
    uint32_t ng = 0;
#pragma unroll
    for (int l = 3 * g; l < 3 * g + 3 && l < kOzP; ++l) ng += __byte_perm(w[l], 0u, 0x4440 | j) * c_oz.gw[l];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] += (uint64_t)ng * c_oz.W[g][i];
    f = fmaf(__uint2float_rn(ng), c_oz.qinv[g], f);
  }
  // f = 16 + sum_l c_l / p_l to about 2^-18, within 1/3 of the multiple of P to
  // take off; |c_l| <= p_l / 2 + 1% keeps it between 7 and 25
  const uint32_t k = (uint32_t)__float2int_rn(f);
#pragma unroll
  for (int i = 0; i < 5; ++i) acc[i] += (uint64_t)k * c_oz.negP[i];
  uint32_t x[5];
  uint64_t c = 0;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    c += acc[i];
    x[i] = (uint32_t)c;
    c >>= 32;
  }
  // sign and magnitude
  const bool neg = (int32_t)x[4] < 0;
  uint64_t lo = (uint64_t)x[1] << 32 | x[0], mid = (uint64_t)x[3] << 32 | x[2];
  uint32_t hi = x[4];
  if (neg) {
    lo = ~lo + 1;
    mid = ~mid + (lo == 0 ? 1 : 0);
    hi = ~hi + ((lo | mid) == 0 ? 1u : 0u);
  }
  // the leading 64 bits from the top nonzero word on, and what lies below them
  uint64_t top, next;
  uint32_t rest = 0;
  int pos;
  if (hi != 0) {
    top = (uint64_t)hi << 32 | (mid >> 32);
    next = mid << 32 | lo >> 32;
    rest = (uint32_t)lo;
    pos = 159;
  } else if (mid != 0) {
    top = mid;
    next = lo;
    pos = 127;
  } else {
    top = lo;
    next = 0;
    pos = 63;
  }
  if (top == 0) return 0.0;
  const int z = __clzll((long long)top);
  const uint64_t mant = z != 0 ? top << z | next >> (64 - z) : top;
  const bool sticky = ((next << z) | rest) != 0;
  uint64_t r = mant >> 11;
  const uint32_t rem = (uint32_t)mant & 0x7ffu;
  if (rem > 0x400u || (rem == 0x400u && (sticky || (r & 1) != 0))) ++r;
  const int e = pos - z + shift;  // exponent of the leading bit
  double y;
  if (e >= -1022 && e <= 1022)
    y = __longlong_as_double((long long)(((uint64_t)(e + 1022) << 52) + r));  // r's bit 52 (or 53) carries in
  else
    y = ldexp((double)r, e - 52);
  return neg ? -y : y;
}

}  // namespace
