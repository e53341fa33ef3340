// Splitting a scalar by the curve's endomorphism: k = k1 + k2 lambda mod n with k1 and
// k2 of half the length, so that k P = k1 P + k2 (beta x, y) takes half the doublings
// (Gallant, Lambert and Vanstone, CRYPTO 2001).  Constants and their derivation are in
// gen_curves.py; only curves of cofactor 1 have them.
#pragma once
#include <cstdint>

#include "curves_gen.cuh"

namespace ecc {

// words 10 .. 14 of k g + 2^319: round(k g / 2^320)
template <class C, bool SECOND>
ECC_DEV void glv_round(uint32_t* c, const uint32_t* k) {
  uint32_t t[15];
#pragma unroll
  for (int i = 0; i < 15; ++i) t[i] = i == 9 ? 0x80000000u : 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    uint64_t carry = 0;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      const uint64_t v = (uint64_t)k[i] * (SECOND ? C::glv_g2(j) : C::glv_g1(j)) + t[i + j] + carry;
      t[i + j] = (uint32_t)v;
      carry = v >> 32;
    }
#pragma unroll
    for (int j = i + 7; j < 15; ++j) {
      carry += t[j];
      t[j] = (uint32_t)carry;
      carry >>= 32;
    }
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) c[i] = t[10 + i];
}

// r += c f mod 2^160, f one of the constants
#define ECC_GLV_MAC(r, c, f)                                         \
  _Pragma("unroll") for (int i = 0; i < 5; ++i) {                    \
    uint64_t carry = 0;                                              \
    _Pragma("unroll") for (int j = 0; i + j < 5; ++j) {              \
      const uint64_t v = (uint64_t)(c)[i] * (f)(j) + (r)[i + j] + carry; \
      (r)[i + j] = (uint32_t)v;                                      \
      carry = v >> 32;                                               \
    }                                                                \
  }

// |v| of a 160-bit two's complement value; returns its sign
ECC_DEV bool glv_abs(uint32_t* v) {
  const bool neg = (v[4] >> 31) != 0;
  uint64_t carry = neg ? 1u : 0u;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    carry += neg ? ~v[i] : v[i];
    v[i] = (uint32_t)carry;
    carry >>= 32;
  }
  return neg;
}

// k < n -> magnitudes m1, m2 (five words, below 2^GLV_BITS) and signs
template <class C>
ECC_DEV void glv_split(const uint32_t* k, uint32_t* m1, bool& neg1, uint32_t* m2, bool& neg2) {
  uint32_t c1[5], c2[5];
  glv_round<C, false>(c1, k);
  glv_round<C, true>(c2, k);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    m1[i] = k[i];
    m2[i] = 0;
  }
  ECC_GLV_MAC(m1, c1, C::glv_a1)
  ECC_GLV_MAC(m1, c2, C::glv_a2)
  ECC_GLV_MAC(m2, c1, C::glv_b1)
  ECC_GLV_MAC(m2, c2, C::glv_b2)
  neg1 = glv_abs(m1);
  neg2 = glv_abs(m2);
}

#undef ECC_GLV_MAC

}  // namespace ecc
