// Prime-field arithmetic on 32-bit limbs (modular arithmetic layer, Section 4).
//
// Elements are N little-endian 32-bit limbs (N even: 8 for 254/256-bit fields,
// 12 for the 381-bit field) held in registers, in Montgomery form a*R mod q,
// canonical in [0, q), with R = 2^(32N), except that the secp256k1 base field
// (FORM 2) is held as plain integers (R = 1).  A field is a traits class F with
//   N, qinv() = -q^-1 mod 2^32, qinv62() = q^-1 mod 2^62, FORM (0 generic, 1 the
//   P-256 prime, 2 the secp256k1 prime, 3 the SM2 prime), p(i),
//   r2(i) = R^2 mod q, r3(i) = R^3 mod q, one(i) = R mod q, pm2(i) = q - 2.
//
// FORM 1-3 multiply as a full 512-bit product (mul_wide8, sqr_wide8) followed by
// a reduction that uses the shape of the prime (Section 4.2): additions only for
// P-256 and SM2, one row of 977 h_i products for secp256k1.  The multiply-add
// pipe takes one warp instruction per 4 cycles, so the 64 (73) wide multiply-adds
// instead of 136 set the time, and the additions run on the other integer pipe
// beside them.  GB300, 16 warps per SM, G modmul/s against the generic product:
// P-256 113 against 68, secp256k1 110 against 68, SM2 107 against 68; squarings
// (36 products instead of 64) 136, 143 and 132; one warp alone takes 245 ns
// instead of 420 (178 for a squaring).
//
// The generic mont_mul is Montgomery multiplication (Algorithm 2) with the operand-scanning
// order interleaved row by row.  Each row A*b_i is split into an "even" chain
// (a_j b_i, j even) and an "odd" chain (a_j b_i, j odd), the mad_n carry chains
// of Section 4.1: within one chain the 64-bit products sit on disjoint word
// pairs, so one chain of alternating mad.lo / mad.hi links covers the row with a
// single carry.  The running value is kept as T = c + 2^32 d with c collecting
// the even chains and d the odd chains; the reduction row u*q (u = T_0 * QINV)
// is split the same way.  Dividing T by 2^32 then only renames registers
// (d becomes the new c, the upper words of c the new d) plus one add for word 0,
// whose carry enters the next odd chain as its carry-in -- so the count is
// 2N^2 + N multiply-adds (136 IMAD.WIDE-class for N = 8), as Section 4.1
// derives, and only ~4N extra adds.  The final value is < 2q and is brought
// into [0, q) with one conditional subtraction.
#pragma once
#include <cstdint>

#include "inv.cuh"
#include "ptx.cuh"

namespace ecc {

template <class F>
struct Fe {
  uint32_t v[F::N];
};

template <class F>
ECC_DEV void fe_copy(uint32_t* r, const uint32_t* a) {
#pragma unroll
  for (int i = 0; i < F::N; ++i) r[i] = a[i];
}

template <class F>
ECC_DEV void fe_set_one(uint32_t* r) {
#pragma unroll
  for (int i = 0; i < F::N; ++i) r[i] = F::one(i);
}

template <class F>
ECC_DEV void fe_set_zero(uint32_t* r) {
#pragma unroll
  for (int i = 0; i < F::N; ++i) r[i] = 0;
}

template <class F>
ECC_DEV bool fe_is_zero(const uint32_t* a) {
  uint32_t acc = 0;
#pragma unroll
  for (int i = 0; i < F::N; ++i) acc |= a[i];
  return acc == 0;
}

template <class F>
ECC_DEV bool fe_eq(const uint32_t* a, const uint32_t* b) {
  uint32_t acc = 0;
#pragma unroll
  for (int i = 0; i < F::N; ++i) acc |= a[i] ^ b[i];
  return acc == 0;
}

// a < q as plain integers (used to validate canonical inputs)
template <class F>
ECC_DEV bool fe_lt_modulus(const uint32_t* a) {
  uint32_t t = ptx::sub_cc(a[0], F::p(0));
#pragma unroll
  for (int i = 1; i < F::N; ++i) t = ptx::subc_cc(a[i], F::p(i));
  uint32_t borrow = ptx::subc(0, 0);
  (void)t;
  return borrow != 0;
}

// r = a + b mod q
template <class F>
ECC_DEV void fe_add(uint32_t* r, const uint32_t* a, const uint32_t* b) {
  constexpr int N = F::N;
  uint32_t t[N], s[N];
  t[0] = ptx::add_cc(a[0], b[0]);
#pragma unroll
  for (int i = 1; i < N; ++i) t[i] = ptx::addc_cc(a[i], b[i]);
  uint32_t top = ptx::addc(0, 0);
  s[0] = ptx::sub_cc(t[0], F::p(0));
#pragma unroll
  for (int i = 1; i < N; ++i) s[i] = ptx::subc_cc(t[i], F::p(i));
  top = ptx::subc(top, 0);  // 0xffffffff iff a + b < q
#pragma unroll
  for (int i = 0; i < N; ++i) r[i] = top ? t[i] : s[i];
}

// r = a - b mod q
template <class F>
ECC_DEV void fe_sub(uint32_t* r, const uint32_t* a, const uint32_t* b) {
  constexpr int N = F::N;
  uint32_t t[N];
  t[0] = ptx::sub_cc(a[0], b[0]);
#pragma unroll
  for (int i = 1; i < N; ++i) t[i] = ptx::subc_cc(a[i], b[i]);
  uint32_t mask = ptx::subc(0, 0);  // 0xffffffff iff a < b
  r[0] = ptx::add_cc(t[0], F::p(0) & mask);
#pragma unroll
  for (int i = 1; i < N - 1; ++i) r[i] = ptx::addc_cc(t[i], F::p(i) & mask);
  r[N - 1] = ptx::addc(t[N - 1], F::p(N - 1) & mask);
}

template <class F>
ECC_DEV void fe_neg(uint32_t* r, const uint32_t* a) {
  uint32_t z[F::N];
  fe_set_zero<F>(z);
  fe_sub<F>(r, z, a);
}

// T = a * b, 16 words.  Products on even words go to E, on odd words to O (the
// mad_n chains of Section 4.1), so each row is one 4-product chain per array; a
// row's carry out either meets a fresh word pair, where product plus carry
// cannot overflow, or is caught in ec / oc and enters the next row's fresh pair.
ECC_DEV void mul_wide8(uint32_t* T, const uint32_t* a, const uint32_t* b) {
  uint32_t E[16], O[16];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const uint64_t e = (uint64_t)a[j] * b[0], o = (uint64_t)a[j + 1] * b[0];
    E[j] = (uint32_t)e;
    E[j + 1] = (uint32_t)(e >> 32);
    O[j + 1] = (uint32_t)o;
    O[j + 2] = (uint32_t)(o >> 32);
  }
  uint32_t ec = 0, oc = 0;
#pragma unroll
  for (int i = 1; i < 8; ++i) {
    uint32_t* const F = (i & 1) ? E : O;  // takes a_1, a_3, a_5, a_7 (top pair fresh)
    uint32_t* const H = (i & 1) ? O : E;  // takes a_0, a_2, a_4, a_6 (carry out to come)
    F[i + 1] = ptx::mad_lo_cc(a[1], b[i], F[i + 1]);
    F[i + 2] = ptx::madc_hi_cc(a[1], b[i], F[i + 2]);
    F[i + 3] = ptx::madc_lo_cc(a[3], b[i], F[i + 3]);
    F[i + 4] = ptx::madc_hi_cc(a[3], b[i], F[i + 4]);
    F[i + 5] = ptx::madc_lo_cc(a[5], b[i], F[i + 5]);
    F[i + 6] = ptx::madc_hi_cc(a[5], b[i], F[i + 6]);
    F[i + 7] = ptx::madc_lo_cc(a[7], b[i], (i & 1) ? ec : oc);
    F[i + 8] = ptx::madc_hi(a[7], b[i], 0);
    H[i] = ptx::mad_lo_cc(a[0], b[i], H[i]);
    H[i + 1] = ptx::madc_hi_cc(a[0], b[i], H[i + 1]);
    H[i + 2] = ptx::madc_lo_cc(a[2], b[i], H[i + 2]);
    H[i + 3] = ptx::madc_hi_cc(a[2], b[i], H[i + 3]);
    H[i + 4] = ptx::madc_lo_cc(a[4], b[i], H[i + 4]);
    H[i + 5] = ptx::madc_hi_cc(a[4], b[i], H[i + 5]);
    H[i + 6] = ptx::madc_lo_cc(a[6], b[i], H[i + 6]);
    H[i + 7] = ptx::madc_hi_cc(a[6], b[i], H[i + 7]);
    ((i & 1) ? oc : ec) = ptx::addc(0, 0);
  }
  // E holds words 0..15, O words 1..14 and its last carry at word 15
  T[0] = E[0];
  T[1] = ptx::add_cc(E[1], O[1]);
#pragma unroll
  for (int k = 2; k < 15; ++k) T[k] = ptx::addc_cc(E[k], O[k]);
  T[15] = ptx::addc(E[15], oc);
}

// T = a^2, 16 words: the 28 products a_i a_j, i < j, once (E and O as above),
// doubled by a shift, plus the 8 squares as one chain.
ECC_DEV void sqr_wide8(uint32_t* T, const uint32_t* a) {
  uint32_t E[16], O[16];
#pragma unroll
  for (int j = 1; j < 8; ++j) {  // row 0: a_0 a_j at word j
    const uint64_t w = (uint64_t)a[0] * a[j];
    uint32_t* const A = (j & 1) ? O : E;
    A[j] = (uint32_t)w;
    A[j + 1] = (uint32_t)(w >> 32);
  }
  E[8] = 0;
  O[9] = 0;
#pragma unroll
  for (int i = 1; i < 7; ++i) {
    // a_i a_j at words i + j: first j = i + 1, i + 3, .. (odd words), then
    // j = i + 2, i + 4, .. (even words).  The chain that ends with a_7 meets a
    // fresh top pair (its low word may hold the other row's caught carry).
#pragma unroll
    for (int par = 1; par <= 2; ++par) {
      uint32_t* const A = par == 1 ? O : E;
      const int last = ((7 - i - par) & 1) ? 6 : 7;
      if (last < i + par) continue;
#pragma unroll
      for (int j = i + par; j <= last; j += 2) {
        const int w = i + j;
        A[w] = j == i + par ? ptx::mad_lo_cc(a[i], a[j], A[w]) : ptx::madc_lo_cc(a[i], a[j], A[w]);
        A[w + 1] = j == 7 ? ptx::madc_hi(a[i], a[j], 0) : ptx::madc_hi_cc(a[i], a[j], A[w + 1]);
      }
      if (last == 6) A[i + 8] = ptx::addc(0, 0);
    }
  }
  uint32_t D[16];
  D[1] = O[1];
  D[2] = ptx::add_cc(E[2], O[2]);
#pragma unroll
  for (int k = 3; k < 14; ++k) D[k] = ptx::addc_cc(E[k], O[k]);
  D[14] = ptx::addc_cc(O[14], 0);
  D[15] = ptx::addc(0, 0);
  uint32_t S[16];
  S[0] = 0;
  S[1] = D[1] << 1;
#pragma unroll
  for (int k = 2; k < 16; ++k) S[k] = __funnelshift_l(D[k - 1], D[k], 1);
  T[0] = ptx::mad_lo_cc(a[0], a[0], S[0]);
  T[1] = ptx::madc_hi_cc(a[0], a[0], S[1]);
#pragma unroll
  for (int k = 1; k < 7; ++k) {
    T[2 * k] = ptx::madc_lo_cc(a[k], a[k], S[2 * k]);
    T[2 * k + 1] = ptx::madc_hi_cc(a[k], a[k], S[2 * k + 1]);
  }
  T[14] = ptx::madc_lo_cc(a[7], a[7], S[14]);
  T[15] = ptx::madc_hi(a[7], a[7], S[15]);
}

// r = t mod q for t < 2q (t: N + 1 words)
template <class F>
ECC_DEV void fe_sub_once(uint32_t* r, const uint32_t* t) {
  constexpr int N = F::N;
  uint32_t s[N];
  s[0] = ptx::sub_cc(t[0], F::p(0));
#pragma unroll
  for (int k = 1; k < N; ++k) s[k] = ptx::subc_cc(t[k], F::p(k));
  const uint32_t top = ptx::subc(t[N], 0);  // 0xffffffff iff t < q
#pragma unroll
  for (int k = 0; k < N; ++k) r[k] = top == 0xffffffffu ? t[k] : s[k];
}

// T R^-1 mod p for p = 2^256 - 2^224 + 2^192 + 2^96 - 1 (NIST P-256), T < p 2^256,
// destroying T.  p = -1 mod 2^96, so u = T mod 2^96 clears 96 bits at a time:
// (T + u p) / 2^96 = (T >> 96) + u + 2^96 W with W = u (1 - 2^32 + 2^64), five
// words that follow u's three without overlap, so a step is W (7 additions) and
// one 8-word chain; a chain's carry has the weight of the next step's third word
// of W and enters there.  Two 96-bit steps and one of 64 bits: 43 additions.
template <class F>
ECC_DEV void redc_p256(uint32_t* r, uint32_t* T) {
  uint32_t W1, W2, W3, W4, x2, x3, x4;
#pragma unroll
  for (int k = 0; k < 6; k += 3) {
    const uint32_t u0 = T[k], u1 = T[k + 1], u2 = T[k + 2];
    x2 = k == 0 ? ptx::add_cc(u2, u0) : ptx::addc_cc(u2, u0);  // carry of the first step
    x3 = ptx::addc_cc(u1, 0);
    x4 = ptx::addc(u2, 0);
    W1 = ptx::sub_cc(u1, u0);
    W2 = ptx::subc_cc(x2, u1);
    W3 = ptx::subc_cc(x3, u2);
    W4 = ptx::subc(x4, 0);
    T[k + 3] = ptx::add_cc(T[k + 3], u0);
    T[k + 4] = ptx::addc_cc(T[k + 4], u1);
    T[k + 5] = ptx::addc_cc(T[k + 5], u2);
    T[k + 6] = ptx::addc_cc(T[k + 6], u0);
    T[k + 7] = ptx::addc_cc(T[k + 7], W1);
    T[k + 8] = ptx::addc_cc(T[k + 8], W2);
    T[k + 9] = ptx::addc_cc(T[k + 9], W3);
    T[k + 10] = ptx::addc_cc(T[k + 10], W4);
  }
  // u = T mod 2^64: T >> 64 plus 2^32 u + 2^128 u (1 - 2^32 + 2^64)
  const uint32_t u0 = T[6], u1 = T[7];
  x2 = ptx::addc_cc(u0, 0);  // carry of the second step
  x3 = ptx::addc(u1, 0);
  W1 = ptx::sub_cc(u1, u0);
  W2 = ptx::subc_cc(x2, u1);
  W3 = ptx::subc(x3, 0);
  uint32_t t[9];
  t[0] = T[8];
  t[1] = ptx::add_cc(T[9], u0);
  t[2] = ptx::addc_cc(T[10], u1);
  t[3] = ptx::addc_cc(T[11], 0);
  t[4] = ptx::addc_cc(T[12], u0);
  t[5] = ptx::addc_cc(T[13], W1);
  t[6] = ptx::addc_cc(T[14], W2);
  t[7] = ptx::addc_cc(T[15], W3);
  t[8] = ptx::addc(0, 0);
  fe_sub_once<F>(r, t);
}

// T mod p for p = 2^256 - 2^32 - 977 (secp256k1), any 512-bit T.  With
// T = lo + 2^256 hi the value is lo + 977 hi + 2^32 hi mod p: the products
// 977 h_i for even i go onto lo, those for odd i onto 2^32 hi (each product pair
// on words that the array already holds), so the fold is 8 wide multiply-adds
// and one merge.  The words above 2^256 (below 2^34) fold once more.
template <class F>
ECC_DEV void red_secp256k1(uint32_t* r, const uint32_t* T) {
  const uint32_t* h = T + 8;
  constexpr uint32_t C = 977u;
  uint32_t e[9], o[10];
  e[0] = ptx::mad_lo_cc(h[0], C, T[0]);
  e[1] = ptx::madc_hi_cc(h[0], C, T[1]);
#pragma unroll
  for (int k = 2; k < 8; k += 2) {
    e[k] = ptx::madc_lo_cc(h[k], C, T[k]);
    e[k + 1] = ptx::madc_hi_cc(h[k], C, T[k + 1]);
  }
  e[8] = ptx::addc(0, 0);
  o[1] = ptx::mad_lo_cc(h[1], C, h[0]);
  o[2] = ptx::madc_hi_cc(h[1], C, h[1]);
#pragma unroll
  for (int k = 3; k < 9; k += 2) {
    o[k] = ptx::madc_lo_cc(h[k], C, h[k - 1]);
    o[k + 1] = ptx::madc_hi_cc(h[k], C, h[k]);
  }
  o[9] = ptx::addc(0, 0);
  e[1] = ptx::add_cc(e[1], o[1]);
#pragma unroll
  for (int k = 2; k < 9; ++k) e[k] = ptx::addc_cc(e[k], o[k]);
  const uint32_t g = ptx::addc(o[9], 0);
  // (e_8 + 2^32 g)(2^32 + 977), g <= 1
  const uint64_t w = (uint64_t)e[8] * C;
  uint32_t x1 = ptx::add_cc((uint32_t)(w >> 32), e[8]);
  uint32_t x2 = ptx::addc(g, 0);
  x1 = ptx::add_cc(x1, g * C);
  x2 = ptx::addc(x2, 0);
  uint32_t t[8], s[8];
  t[0] = ptx::add_cc(e[0], (uint32_t)w);
  t[1] = ptx::addc_cc(e[1], x1);
  t[2] = ptx::addc_cc(e[2], x2);
#pragma unroll
  for (int k = 3; k < 8; ++k) t[k] = ptx::addc_cc(e[k], 0);
  uint32_t over = ptx::addc(0, 0);
  // t + 2^256 over < 2p: t + 2^32 + 977 carries, or over is set, iff it is >= p
  s[0] = ptx::add_cc(t[0], C);
  s[1] = ptx::addc_cc(t[1], 1u);
#pragma unroll
  for (int k = 2; k < 8; ++k) s[k] = ptx::addc_cc(t[k], 0);
  over = ptx::addc(over, 0);
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = over ? s[k] : t[k];
}

// T R^-1 mod p for p = 2^256 - 2^224 - 2^96 + 2^64 - 1 (SM2), T < p 2^256.  With
// m = T_lo (-p^-1) mod 2^256 the result is (T + m p) / 2^256, and both parts are
// additions of shifted m:
//   m = T_lo + (m << 64) - (m << 96) - (m << 224) mod 2^256 (word by word; the
//       carry of the sum and the two borrows are the low part's carry),
//   r = T_hi + m + (m >> 192) - (m >> 160) - (m >> 32) + carry - borrows.
// 55 additions, against 88 for four 64-bit steps (107 against 75-85 G modmul/s).
template <class F>
ECC_DEV void redc_sm2(uint32_t* r, const uint32_t* T) {
  uint32_t m[8], A[8], c, b;
  m[0] = T[0];
  m[1] = T[1];
  m[2] = ptx::add_cc(T[2], m[0]);
  A[3] = ptx::addc_cc(T[3], m[1]);
  A[4] = ptx::addc_cc(T[4], m[2]);
  c = ptx::addc(0, 0);
  m[3] = ptx::sub_cc(A[3], m[0]);
  m[4] = ptx::subc_cc(A[4], m[1]);
  b = ptx::subc(0, 0);
  ptx::add_cc(c, 0xffffffffu);  // restores the carry (a borrow: 0 - b below)
  A[5] = ptx::addc_cc(T[5], m[3]);
  A[6] = ptx::addc_cc(T[6], m[4]);
  c = ptx::addc(0, 0);
  ptx::sub_cc(0, b);
  m[5] = ptx::subc_cc(A[5], m[2]);
  m[6] = ptx::subc_cc(A[6], m[3]);
  b = ptx::subc(0, 0);
  ptx::add_cc(c, 0xffffffffu);
  A[7] = ptx::addc_cc(T[7], m[5]);
  c = ptx::addc(0, 0);  // carry of the low part
  ptx::sub_cc(0, b);
  m[7] = ptx::subc_cc(A[7], m[4]);
  b = ptx::subc(0, 0);  // its first borrow
  m[7] = ptx::sub_cc(m[7], m[0]);
  const uint32_t b2 = ptx::subc(0, 0);  // its second borrow
  // S = (m >> 32) + (m >> 160) - (m >> 192) + second borrow
  uint32_t S[8], t[9];
  const uint32_t d0 = ptx::sub_cc(m[5], m[6]);
  const uint32_t d1 = ptx::subc_cc(m[6], m[7]);
  const uint32_t d2 = ptx::subc(m[7], 0);
  ptx::add_cc(b2, 1u);  // carries iff b2 is all ones
  S[0] = ptx::addc_cc(m[1], d0);
  S[1] = ptx::addc_cc(m[2], d1);
  S[2] = ptx::addc_cc(m[3], d2);
#pragma unroll
  for (int k = 3; k < 7; ++k) S[k] = ptx::addc_cc(m[k + 1], 0);
  S[7] = ptx::addc(0, 0);
  ptx::add_cc(c, 0xffffffffu);
#pragma unroll
  for (int k = 0; k < 8; ++k) t[k] = ptx::addc_cc(T[8 + k], m[k]);
  t[8] = ptx::addc(0, 0);
  ptx::sub_cc(0, b);
#pragma unroll
  for (int k = 0; k < 8; ++k) t[k] = ptx::subc_cc(t[k], S[k]);
  t[8] = ptx::subc(t[8], 0);
  fe_sub_once<F>(r, t);
}

// The reduction of a 512-bit product for FORM 1-3 (T is destroyed).
template <class F>
ECC_DEV void reduce_wide(uint32_t* r, uint32_t* T) {
  static_assert(F::FORM >= 1 && F::FORM <= 3 && F::N == 8, "special-form primes");
  if constexpr (F::FORM == 1) {
    redc_p256<F>(r, T);
  } else if constexpr (F::FORM == 2) {
    red_secp256k1<F>(r, T);
  } else {
    redc_sm2<F>(r, T);
  }
}

// Montgomery product r = a * b * R^-1 mod q (r may alias a or b).
template <class F>
ECC_DEV void mont_mul(uint32_t* r, const uint32_t* a, const uint32_t* b) {
  constexpr int N = F::N;
  static_assert(N % 2 == 0, "even limb count");
  if constexpr (F::FORM != 0) {
    uint32_t T[16];
    mul_wide8(T, a, b);
    reduce_wide<F>(r, T);
    return;
  }
  uint32_t c[N + 1], d[N + 1];
#pragma unroll
  for (int i = 0; i < N + 1; ++i) {
    c[i] = 0;
    d[i] = 0;
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t bi = b[i];
    if (i == 0) {
      // odd chain: d[j-1], d[j] += a_j * b_0 for odd j
      d[0] = ptx::mad_lo_cc(a[1], bi, d[0]);
      d[1] = ptx::madc_hi_cc(a[1], bi, d[1]);
    } else {
      // T /= 2^32: new c = (d0 + c1, d1, .., dN), new d = (c2, .., cN, 0, 0);
      // the carry of d0 + c1 (word 1) is the carry-in of the odd chain.
      uint32_t nc0 = ptx::add_cc(d[0], c[1]);
#pragma unroll
      for (int k = 0; k < N - 1; ++k) {
        uint32_t t = d[k + 1];
        d[k] = c[k + 2];
        c[k + 1] = t;
      }
      c[N] = d[N];
      c[0] = nc0;
      d[N - 1] = 0;
      d[N] = 0;
      d[0] = ptx::madc_lo_cc(a[1], bi, d[0]);
      d[1] = ptx::madc_hi_cc(a[1], bi, d[1]);
    }
#pragma unroll
    for (int j = 3; j < N; j += 2) {
      d[j - 1] = ptx::madc_lo_cc(a[j], bi, d[j - 1]);
      d[j] = ptx::madc_hi_cc(a[j], bi, d[j]);
    }
    d[N] = ptx::addc(d[N], 0);
    // even chain: c[j], c[j+1] += a_j * b_i for even j
    c[0] = ptx::mad_lo_cc(a[0], bi, c[0]);
    c[1] = ptx::madc_hi_cc(a[0], bi, c[1]);
#pragma unroll
    for (int j = 2; j < N; j += 2) {
      c[j] = ptx::madc_lo_cc(a[j], bi, c[j]);
      c[j + 1] = ptx::madc_hi_cc(a[j], bi, c[j + 1]);
    }
    c[N] = ptx::addc(c[N], 0);
    // reduction row: u = T_0 * QINV, T += u * q (even and odd chains)
    const uint32_t u = c[0] * F::qinv();
    c[0] = ptx::mad_lo_cc(u, F::p(0), c[0]);
    c[1] = ptx::madc_hi_cc(u, F::p(0), c[1]);
#pragma unroll
    for (int j = 2; j < N; j += 2) {
      c[j] = ptx::madc_lo_cc(u, F::p(j), c[j]);
      c[j + 1] = ptx::madc_hi_cc(u, F::p(j), c[j + 1]);
    }
    c[N] = ptx::addc(c[N], 0);
    d[0] = ptx::mad_lo_cc(u, F::p(1), d[0]);
    d[1] = ptx::madc_hi_cc(u, F::p(1), d[1]);
#pragma unroll
    for (int j = 3; j < N; j += 2) {
      d[j - 1] = ptx::madc_lo_cc(u, F::p(j), d[j - 1]);
      d[j] = ptx::madc_hi_cc(u, F::p(j), d[j]);
    }
    d[N] = ptx::addc(d[N], 0);
  }
  // last division by 2^32 and merge: t = d + (c >> 32 bits), t < 2q
  uint32_t t[N + 1];
  t[0] = ptx::add_cc(d[0], c[1]);
#pragma unroll
  for (int k = 1; k < N; ++k) t[k] = ptx::addc_cc(d[k], c[k + 1]);
  t[N] = ptx::addc(d[N], 0);
  fe_sub_once<F>(r, t);
}

// r = a^2 R^-1 mod q for q < 2^(32 N - 1), rows as in mont_mul: row i adds only
// a_i^2 and 2 a_i a_j, j > i, so it has N - i products and its lowest word is i; the
// reduction row of word 0 can go first.  N (N + 1) / 2 + N^2 + N multiply-adds (108 of
// 136 with 8 limbs, 234 of 300 with 12) in as many registers as mont_mul.
template <class F>
ECC_DEV void mont_sqr_rows(uint32_t* r, const uint32_t* a) {
  constexpr int N = F::N;
  uint32_t c[N + 1], d[N + 1], a2[N];  // a2: limbs of 2 a
#pragma unroll
  for (int i = 0; i < N + 1; ++i) c[i] = d[i] = 0;
#pragma unroll
  for (int i = 1; i < N; ++i) a2[i] = __funnelshift_l(a[i - 1], a[i], 1);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    // the row's factor of a_i at word j >= i: 2 (a >> 32 (i + 1)) has no bit of a_i
    auto f = [&](int j) { return j == i ? a[i] : j == i + 1 ? a[j] << 1 : a2[j]; };
    auto row = [&]() {
      const int o = i | 1, e = (i + 1) & ~1;  // first odd and even word
#pragma unroll
      for (int j = o; j < N; j += 2) {
        d[j - 1] = j == o ? ptx::mad_lo_cc(f(j), a[i], d[j - 1]) : ptx::madc_lo_cc(f(j), a[i], d[j - 1]);
        d[j] = ptx::madc_hi_cc(f(j), a[i], d[j]);
      }
      d[N] = ptx::addc(d[N], 0);
      if (e < N) {
#pragma unroll
        for (int j = e; j < N; j += 2) {
          c[j] = j == e ? ptx::mad_lo_cc(f(j), a[i], c[j]) : ptx::madc_lo_cc(f(j), a[i], c[j]);
          c[j + 1] = ptx::madc_hi_cc(f(j), a[i], c[j + 1]);
        }
        c[N] = ptx::addc(c[N], 0);
      }
    };
    uint32_t u;
    if (i == 0) {
      row();
      u = c[0] * F::qinv();
      d[0] = ptx::mad_lo_cc(u, F::p(1), d[0]);
    } else {  // T /= 2^32; the carry of d0 + c1 enters the odd reduction chain
      const uint32_t nc0 = ptx::add_cc(d[0], c[1]);
#pragma unroll
      for (int k = 0; k < N - 1; ++k) {
        const uint32_t t = d[k + 1];
        d[k] = c[k + 2];
        c[k + 1] = t;
      }
      c[N] = d[N];
      c[0] = nc0;
      d[N - 1] = 0;
      d[N] = 0;
      u = nc0 * F::qinv();
      d[0] = ptx::madc_lo_cc(u, F::p(1), d[0]);
    }
    d[1] = ptx::madc_hi_cc(u, F::p(1), d[1]);
#pragma unroll
    for (int j = 3; j < N; j += 2) {
      d[j - 1] = ptx::madc_lo_cc(u, F::p(j), d[j - 1]);
      d[j] = ptx::madc_hi_cc(u, F::p(j), d[j]);
    }
    d[N] = ptx::addc(d[N], 0);
    c[0] = ptx::mad_lo_cc(u, F::p(0), c[0]);
    c[1] = ptx::madc_hi_cc(u, F::p(0), c[1]);
#pragma unroll
    for (int j = 2; j < N; j += 2) {
      c[j] = ptx::madc_lo_cc(u, F::p(j), c[j]);
      c[j + 1] = ptx::madc_hi_cc(u, F::p(j), c[j + 1]);
    }
    c[N] = ptx::addc(c[N], 0);
    if (i > 0) row();
  }
  uint32_t t[N + 1];
  t[0] = ptx::add_cc(d[0], c[1]);
#pragma unroll
  for (int k = 1; k < N; ++k) t[k] = ptx::addc_cc(d[k], c[k + 1]);
  t[N] = ptx::addc(d[N], 0);
  fe_sub_once<F>(r, t);
}

// r = (a b + x y) R^-1 mod q for q < R / 4 with one reduction (2 N^2 + N^2 + N
// multiply-adds instead of 4 N^2 + 2 N): the sum is below 2 q R / 4 + q R, so one
// subtraction is enough.
template <class F>
ECC_DEV void mont_mul2(uint32_t* r, const uint32_t* a, const uint32_t* b, const uint32_t* x, const uint32_t* y) {
  constexpr int N = F::N;
  static_assert(F::BITS <= 32 * N - 2, "room for the sum");
  uint32_t c[N + 1], d[N + 1];
#pragma unroll
  for (int i = 0; i < N + 1; ++i) c[i] = d[i] = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (i == 0) {
      d[0] = ptx::mad_lo_cc(a[1], b[0], d[0]);
    } else {
      const uint32_t nc0 = ptx::add_cc(d[0], c[1]);
#pragma unroll
      for (int k = 0; k < N - 1; ++k) {
        const uint32_t t = d[k + 1];
        d[k] = c[k + 2];
        c[k + 1] = t;
      }
      c[N] = d[N];
      c[0] = nc0;
      d[N - 1] = 0;
      d[N] = 0;
      d[0] = ptx::madc_lo_cc(a[1], b[i], d[0]);
    }
    d[1] = ptx::madc_hi_cc(a[1], b[i], d[1]);
#pragma unroll
    for (int j = 3; j < N; j += 2) {
      d[j - 1] = ptx::madc_lo_cc(a[j], b[i], d[j - 1]);
      d[j] = ptx::madc_hi_cc(a[j], b[i], d[j]);
    }
    d[N] = ptx::addc(d[N], 0);
#pragma unroll
    for (int j = 1; j < N; j += 2) {
      d[j - 1] = j == 1 ? ptx::mad_lo_cc(x[j], y[i], d[j - 1]) : ptx::madc_lo_cc(x[j], y[i], d[j - 1]);
      d[j] = ptx::madc_hi_cc(x[j], y[i], d[j]);
    }
    d[N] = ptx::addc(d[N], 0);
#pragma unroll
    for (int j = 0; j < N; j += 2) {
      c[j] = j == 0 ? ptx::mad_lo_cc(a[j], b[i], c[j]) : ptx::madc_lo_cc(a[j], b[i], c[j]);
      c[j + 1] = ptx::madc_hi_cc(a[j], b[i], c[j + 1]);
    }
    c[N] = ptx::addc(c[N], 0);
#pragma unroll
    for (int j = 0; j < N; j += 2) {
      c[j] = j == 0 ? ptx::mad_lo_cc(x[j], y[i], c[j]) : ptx::madc_lo_cc(x[j], y[i], c[j]);
      c[j + 1] = ptx::madc_hi_cc(x[j], y[i], c[j + 1]);
    }
    c[N] = ptx::addc(c[N], 0);
    const uint32_t u = c[0] * F::qinv();
#pragma unroll
    for (int j = 0; j < N; j += 2) {
      c[j] = j == 0 ? ptx::mad_lo_cc(u, F::p(j), c[j]) : ptx::madc_lo_cc(u, F::p(j), c[j]);
      c[j + 1] = ptx::madc_hi_cc(u, F::p(j), c[j + 1]);
    }
    c[N] = ptx::addc(c[N], 0);
#pragma unroll
    for (int j = 1; j < N; j += 2) {
      d[j - 1] = j == 1 ? ptx::mad_lo_cc(u, F::p(j), d[j - 1]) : ptx::madc_lo_cc(u, F::p(j), d[j - 1]);
      d[j] = ptx::madc_hi_cc(u, F::p(j), d[j]);
    }
    d[N] = ptx::addc(d[N], 0);
  }
  uint32_t t[N + 1];
  t[0] = ptx::add_cc(d[0], c[1]);
#pragma unroll
  for (int k = 1; k < N; ++k) t[k] = ptx::addc_cc(d[k], c[k + 1]);
  t[N] = ptx::addc(d[N], 0);
  fe_sub_once<F>(r, t);
}

template <class F>
ECC_DEV void mont_sqr(uint32_t* r, const uint32_t* a) {
  if constexpr (F::FORM != 0) {
    uint32_t T[16];
    sqr_wide8(T, a);
    reduce_wide<F>(r, T);
  } else if constexpr (F::SQR_ROWS) {
    mont_sqr_rows<F>(r, a);
  } else {
    mont_mul<F>(r, a, a);
  }
}

// r = a b - c d with one reduction: of the difference of the two products for FORM
// 1-3 (52 additions fewer than two reductions and a subtraction; a negative
// difference gets q 2^256), of a b + (q - c) d for the others.
ECC_DEV bool sub_wide(uint32_t* A, const uint32_t* B) {
  A[0] = ptx::sub_cc(A[0], B[0]);
#pragma unroll
  for (int k = 1; k < 16; ++k) A[k] = ptx::subc_cc(A[k], B[k]);
  return ptx::subc(0, 0) != 0;
}

template <class F>
ECC_DEV void reduce_diff(uint32_t* r, uint32_t* A, const uint32_t* B) {
  const uint32_t mask = sub_wide(A, B) ? 0xffffffffu : 0u;
  A[8] = ptx::add_cc(A[8], F::p(0) & mask);
#pragma unroll
  for (int k = 1; k < 7; ++k) A[8 + k] = ptx::addc_cc(A[8 + k], F::p(k) & mask);
  A[15] = ptx::addc(A[15], F::p(7) & mask);
  reduce_wide<F>(r, A);
}

template <class F>
ECC_DEV void mont_mul_sub(uint32_t* r, const uint32_t* a, const uint32_t* b, const uint32_t* c,
                          const uint32_t* d) {
  if constexpr (F::FORM != 0) {
    uint32_t A[16], B[16];
    mul_wide8(A, a, b);
    mul_wide8(B, c, d);
    reduce_diff<F>(r, A, B);
  } else {
    uint32_t t[F::N];
    fe_neg<F>(t, c);
    mont_mul2<F>(r, a, b, t, d);
  }
}

// r = a b - c^2
template <class F>
ECC_DEV void mont_mul_sub_sqr(uint32_t* r, const uint32_t* a, const uint32_t* b, const uint32_t* c) {
  if constexpr (F::FORM != 0) {
    uint32_t A[16], B[16];
    mul_wide8(A, a, b);
    sqr_wide8(B, c);
    reduce_diff<F>(r, A, B);
  } else {
    uint32_t t[F::N];
    fe_neg<F>(t, c);
    mont_mul2<F>(r, a, b, t, c);
  }
}

// canonical integer -> Montgomery form (a * R^2 * R^-1 = a R)
template <class F>
ECC_DEV void to_mont(uint32_t* r, const uint32_t* a) {
  if constexpr (F::FORM == 2) {  // held as plain integers
    fe_copy<F>(r, a);
    return;
  }
  uint32_t r2[F::N];
#pragma unroll
  for (int i = 0; i < F::N; ++i) r2[i] = F::r2(i);
  mont_mul<F>(r, a, r2);
}

// Montgomery form -> canonical integer
template <class F>
ECC_DEV void from_mont(uint32_t* r, const uint32_t* a) {
  if constexpr (F::FORM == 2) {
    fe_copy<F>(r, a);
    return;
  }
  uint32_t one[F::N];
#pragma unroll
  for (int i = 0; i < F::N; ++i) one[i] = i == 0 ? 1u : 0u;
  mont_mul<F>(r, a, one);
}

// r = a^(q-2) = a^-1 (Fermat, Section 2.2); a = 0 gives 0.  Fixed 4-bit
// windows over the exponent, most significant first.  Used by one thread per
// batch (the "apply" step of the gather-apply-scatter batch inversion).
template <class F>
__device__ __noinline__ void fe_inv_fermat(uint32_t* r, const uint32_t* a) {
  constexpr int N = F::N;
  uint32_t tab[16][N];
  fe_set_one<F>(tab[0]);
  fe_copy<F>(tab[1], a);
  for (int k = 2; k < 16; ++k) mont_mul<F>(tab[k], tab[k - 1], a);
  uint32_t acc[N];
  fe_set_one<F>(acc);
  for (int w = 8 * N - 1; w >= 0; --w) {
    const uint32_t digit = (F::pm2(w >> 3) >> (4 * (w & 7))) & 15u;
    for (int s = 0; s < 4; ++s) mont_sqr<F>(acc, acc);
    uint32_t t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = tab[digit][i];
    mont_mul<F>(acc, acc, t);
  }
  fe_copy<F>(r, acc);
}

// a^-1 mod q as an integer, 0 for 0, by the divstep inversion of inv.cuh on 30-bit
// limbs with branch-free divsteps.  Out of line, operand and result in registers:
// it is the serial step of every batched round.
template <class F, bool FLAT = true>
__device__ __noinline__ Fe<F> fe_inv_call(Fe<F> a) {
  constexpr int N = F::N;
  constexpr int L = (32 * N + 2 + 29) / 30;
  uint32_t q[N], x[N];
#pragma unroll
  for (int i = 0; i < N; ++i) q[i] = F::p(i);
  inv_divsteps30<L, N, FLAT>(x, a.v, q, (uint32_t)F::qinv62() & (uint32_t)kM30);
  fe_copy<F>(a.v, x);
  return a;
}

template <class F, bool FLAT = true>
ECC_DEV void fe_inv_int(uint32_t* r, const uint32_t* a) {
  Fe<F> x;
  fe_copy<F>(x.v, a);
  x = fe_inv_call<F, FLAT>(x);
  fe_copy<F>(r, x.v);
}

// r = a^-1 in Montgomery form (a = x R -> r = x^-1 R), a = 0 gives 0: (x R)^-1 on
// the integer, then one Montgomery product with R^3 mod q restores the form.
template <class F, bool FLAT = true>
ECC_DEV void fe_inv_mont(uint32_t* r, const uint32_t* a) {
  constexpr int N = F::N;
  uint32_t x[N], r3[N];
#pragma unroll
  for (int i = 0; i < N; ++i) r3[i] = F::r3(i);
  fe_inv_int<F, FLAT>(x, a);
  mont_mul<F>(r, x, r3);
}

// The same with the 62-bit-limb divsteps (64 x 64 -> 128-bit products), kept
// for the inversion probe.
template <class F>
__device__ __noinline__ void fe_inv_mont62(uint32_t* r, const uint32_t* a) {
  constexpr int N = F::N;
  constexpr int L = (32 * N + 2 + 61) / 62;
  uint32_t q[N], x[N], r3[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    q[i] = F::p(i);
    r3[i] = F::r3(i);
  }
  inv_divsteps<L>(x, a, q, N, F::qinv62());
  mont_mul<F>(r, x, r3);
}

}  // namespace ecc
