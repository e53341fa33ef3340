// Scalar multiplication by one thread in Jacobian coordinates (x = X/Z^2,
// y = Y/Z^3, Z = 0 for O; Section 2.1.2), used by ECDSA verification, signing and
// FPMUL: the whole chain stays in registers, no thread waits for another, and
// the only inversions are the few at its ends.
//
// Batched affine rounds (Section 3.3) need fewer multiplications per operation (6
// or 7 against 7 to 11), but every round of a scalar multiplication moves the
// batch's state through memory (113 GB for 2^20 verifications) and waits for
// one serial inversion (39 us a round, 314 rounds): with the multiplications of
// fp.cuh the chains in registers are faster at every batch size.  One inversion
// per thread costs no more than one per warp: the branch-free divsteps run all 32
// lanes in the time of one (13.5 against 13.4 us).
#pragma once
#include "ec.cuh"

namespace ecc {

// r = a / 2 mod q
template <class F>
ECC_DEV void fe_half(uint32_t* r, const uint32_t* a) {
  constexpr int N = F::N;
  const uint32_t mask = 0u - (a[0] & 1u);
  uint32_t t[N + 1];
  t[0] = ptx::add_cc(a[0], F::p(0) & mask);
#pragma unroll
  for (int i = 1; i < N; ++i) t[i] = ptx::addc_cc(a[i], F::p(i) & mask);
  t[N] = ptx::addc(0, 0);
#pragma unroll
  for (int i = 0; i < N; ++i) r[i] = __funnelshift_r(t[i], t[i + 1], 1);
}

// Out-of-line products with operands and result in registers.  The addition
// below uses them: written out in full it is 29 KB of code beside the doubling's
// 22 KB, more than the instruction cache holds, and warps at different places of
// the loop then wait for instructions (1.8 of 7.9 cycles an issue).  The 2^20 P-256
// batch took 46.3 ms that way and takes 33.2 with the addition's products called
// and a barrier per operation (below).
template <class F>
__device__ __noinline__ Fe<F> mul_call(Fe<F> a, Fe<F> b) {
  mont_mul<F>(a.v, a.v, b.v);
  return a;
}
template <class F>
__device__ __noinline__ Fe<F> sqr_call(Fe<F> a) {
  mont_sqr<F>(a.v, a.v);
  return a;
}
template <class F>
__device__ __noinline__ Fe<F> mul_sub_call(Fe<F> a, Fe<F> b, Fe<F> c, Fe<F> d) {
  mont_mul_sub<F>(a.v, a.v, b.v, c.v, d.v);
  return a;
}

template <class F>
ECC_DEV Fe<F> fe_pack(const uint32_t* a) {
  Fe<F> x;
  fe_copy<F>(x.v, a);
  return x;
}
template <class F>
ECC_DEV void call_mul(uint32_t* r, const uint32_t* a, const uint32_t* b) {
  const Fe<F> x = mul_call<F>(fe_pack<F>(a), fe_pack<F>(b));
  fe_copy<F>(r, x.v);
}
template <class F>
ECC_DEV void call_sqr(uint32_t* r, const uint32_t* a) {
  const Fe<F> x = sqr_call<F>(fe_pack<F>(a));
  fe_copy<F>(r, x.v);
}
template <class F>
ECC_DEV void call_mul_sub(uint32_t* r, const uint32_t* a, const uint32_t* b, const uint32_t* c,
                          const uint32_t* d) {
  const Fe<F> x = mul_sub_call<F>(fe_pack<F>(a), fe_pack<F>(b), fe_pack<F>(c), fe_pack<F>(d));
  fe_copy<F>(r, x.v);
}

// P <- 2 P.  The usual formulas with every coordinate scaled by Z -> Z / 2: with
// l = (3 X^2 + a Z^4) / 2, X3 = l^2 - 2 X Y^2, Y3 = l (X Y^2 - X3) - Y^4,
// Z3 = Y Z: 4 products and 4 squares (a = -3, 3 X^2 + a Z^4 = 3 (X - Z^2)(X + Z^2)) or
// 3 and 4 (a = 0), and no multiples by 4 or 8.  O stays O.
template <class C>
ECC_DEV void jac_dbl_half(uint32_t* X, uint32_t* Y, uint32_t* Z) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  uint32_t l[N], t[N], YY[N], XYY[N];
  if constexpr (C::A_ZERO) {
    mont_sqr<F>(l, X);
  } else {
    uint32_t u[N];
    mont_sqr<F>(t, Z);
    fe_sub<F>(u, X, t);
    fe_add<F>(t, X, t);
    mont_mul<F>(l, u, t);
  }
  fe_half<F>(t, l);
  fe_add<F>(l, l, t);
  mont_mul<F>(Z, Y, Z);
  mont_sqr<F>(YY, Y);
  mont_mul<F>(XYY, X, YY);
  mont_sqr<F>(X, l);
  fe_sub<F>(X, X, XYY);
  fe_sub<F>(X, X, XYY);
  fe_sub<F>(t, XYY, X);
  mont_mul_sub_sqr<F>(Y, l, t, YY);
}

template <class F>
struct JacReg {
  Fe<F> X, Y, Z;
};

// The doubling inside an addition of equal points (rare), out of line and through
// memory, so that the additions around it keep their registers.
template <class C>
__device__ __noinline__ void jac_dbl_mem(uint32_t* P) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  uint32_t X[N], Y[N], Z[N];
  fe_copy<F>(X, P);
  fe_copy<F>(Y, P + N);
  fe_copy<F>(Z, P + 2 * N);
  jac_dbl_half<C>(X, Y, Z);
  fe_copy<F>(P, X);
  fe_copy<F>(P + N, Y);
  fe_copy<F>(P + 2 * N, Z);
}

template <class C>
ECC_DEV void jac_dbl_rare(uint32_t* X, uint32_t* Y, uint32_t* Z) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  uint32_t P[3 * N];
  fe_copy<F>(P, X);
  fe_copy<F>(P + N, Y);
  fe_copy<F>(P + 2 * N, Z);
  jac_dbl_mem<C>(P);
  fe_copy<F>(X, P);
  fe_copy<F>(Y, P + N);
  fe_copy<F>(Z, P + 2 * N);
}

// P <- P + (x, y) for an affine point other than O; every case of the group law.
// When both operands are finite and x_P != x, Z3 = Z H with H = x Z^2 - X left in
// H (8 products and 3 squares).
template <class C>
ECC_DEV void jac_madd(uint32_t* X, uint32_t* Y, uint32_t* Z, const uint32_t* x, const uint32_t* y,
                      uint32_t* H) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  if (fe_is_zero<F>(Z)) {
    fe_copy<F>(X, x);
    fe_copy<F>(Y, y);
    fe_set_one<F>(Z);
    return;
  }
  uint32_t t[N], r[N];
  call_sqr<F>(t, Z);
  call_mul<F>(H, x, t);
  fe_sub<F>(H, H, X);
  call_mul<F>(t, t, Z);
  call_mul<F>(r, y, t);
  fe_sub<F>(r, r, Y);
  if (fe_is_zero<F>(H)) {
    if (fe_is_zero<F>(r)) {
      jac_dbl_rare<C>(X, Y, Z);
    } else {
      fe_set_zero<F>(Z);
    }
    return;
  }
  uint32_t V[N];
  call_mul<F>(Z, Z, H);
  call_sqr<F>(t, H);
  call_mul<F>(V, X, t);
  call_mul<F>(t, H, t);
  call_sqr<F>(X, r);
  fe_sub<F>(X, X, t);
  fe_sub<F>(X, X, V);
  fe_sub<F>(X, X, V);
  fe_sub<F>(V, V, X);
  call_mul_sub<F>(Y, r, V, Y, t);
}

// ---------------------------------------------------------------- quads
// A group operation by the four lanes of a quad, for chains with too few of them to
// fill the GPU: the lanes hold the same points and take one product each of a
// step's independent ones, so a doubling costs 3 (a = 0) or 4 products' latency and
// an addition of an affine point 5, instead of 7, 8 and 11, plus the exchange of the
// products.  The four lanes call these together with equal operands; other quads of
// the warp may be elsewhere.

ECC_DEV unsigned quad_mask() { return 0xfu << (threadIdx.x & 28u); }

template <class F>
ECC_DEV void quad_get(uint32_t* r, const uint32_t* a, int lane) {
  const unsigned m = quad_mask();
#pragma unroll
  for (int i = 0; i < F::N; ++i) r[i] = __shfl_sync(m, a[i], lane, 4);
}

// this lane's factor: a, b, c or d for lane 0, 1, 2 or 3 of the quad
template <class F>
ECC_DEV void quad_pick(uint32_t* r, const uint32_t* a, const uint32_t* b, const uint32_t* c, const uint32_t* d) {
  const unsigned q = threadIdx.x & 3u;
#pragma unroll
  for (int i = 0; i < F::N; ++i) {
    const uint32_t lo = (q & 1u) ? b[i] : a[i], hi = (q & 1u) ? d[i] : c[i];
    r[i] = (q & 2u) ? hi : lo;
  }
}

// P <- 2 P, the formulas of jac_dbl_half
template <class C>
ECC_DEV void quad_dbl(JacReg<typename C::Fp>& P) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  uint32_t a[N], b[N], p[N], l[N], YY[N], D[N];
  if constexpr (C::A_ZERO) {
    quad_pick<F>(a, P.X.v, P.Y.v, P.Y.v, P.X.v);
    quad_pick<F>(b, P.X.v, P.Y.v, P.Z.v, P.X.v);
    mont_mul<F>(p, a, b);  // X^2, Y^2, Y Z
    quad_get<F>(l, p, 0);
    quad_get<F>(YY, p, 1);
    quad_get<F>(P.Z.v, p, 2);
    fe_half<F>(a, l);
    fe_add<F>(l, l, a);    // 3 X^2 / 2
    quad_pick<F>(a, YY, P.X.v, l, l);
    quad_pick<F>(b, YY, YY, l, l);
    mont_mul<F>(p, a, b);  // Y^4, X Y^2, l^2
  } else {
    quad_pick<F>(a, P.Z.v, P.Y.v, P.Y.v, P.Z.v);
    quad_pick<F>(b, P.Z.v, P.Y.v, P.Z.v, P.Z.v);
    mont_mul<F>(p, a, b);  // Z^2, Y^2, Y Z
    quad_get<F>(l, p, 0);
    quad_get<F>(YY, p, 1);
    quad_get<F>(P.Z.v, p, 2);
    fe_add<F>(D, P.X.v, l);
    fe_sub<F>(l, P.X.v, l);
    quad_pick<F>(a, YY, P.X.v, l, l);
    quad_pick<F>(b, YY, YY, D, D);
    mont_mul<F>(p, a, b);  // Y^4, X Y^2, X^2 - Z^4
    quad_get<F>(l, p, 2);
    fe_half<F>(a, l);
    fe_add<F>(l, l, a);
    mont_mul<F>(a, l, l);  // l^2, in every lane; p keeps the other products
  }
  quad_get<F>(YY, p, 0);
  quad_get<F>(D, p, 1);
  if constexpr (C::A_ZERO) {
    quad_get<F>(P.X.v, p, 2);
  } else {
    fe_copy<F>(P.X.v, a);
  }
  fe_sub<F>(P.X.v, P.X.v, D);
  fe_sub<F>(P.X.v, P.X.v, D);
  fe_sub<F>(D, D, P.X.v);
  mont_mul<F>(P.Y.v, l, D);
  fe_sub<F>(P.Y.v, P.Y.v, YY);
}

// jac_madd by a quad
template <class C>
ECC_DEV void quad_madd(JacReg<typename C::Fp>& P, const uint32_t* x, const uint32_t* y, uint32_t* H) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  if (fe_is_zero<F>(P.Z.v)) {
    fe_copy<F>(P.X.v, x);
    fe_copy<F>(P.Y.v, y);
    fe_set_one<F>(P.Z.v);
    return;
  }
  uint32_t a[N], b[N], p[N], t[N], r[N], V[N];
  quad_pick<F>(a, P.Z.v, y, P.Z.v, y);
  mont_mul<F>(p, a, P.Z.v);  // Z^2, y Z
  quad_get<F>(t, p, 0);
  quad_get<F>(r, p, 1);
  quad_pick<F>(a, x, r, x, r);
  mont_mul<F>(p, a, t);      // x Z^2, y Z^3
  quad_get<F>(H, p, 0);
  fe_sub<F>(H, H, P.X.v);
  quad_get<F>(r, p, 1);
  fe_sub<F>(r, r, P.Y.v);
  if (fe_is_zero<F>(H)) {
    if (fe_is_zero<F>(r)) {
      jac_dbl_rare<C>(P.X.v, P.Y.v, P.Z.v);
    } else {
      fe_set_zero<F>(P.Z.v);
    }
    return;
  }
  quad_pick<F>(a, H, P.Z.v, r, H);
  quad_pick<F>(b, H, H, r, H);
  mont_mul<F>(p, a, b);      // H^2, Z H, r^2
  quad_get<F>(t, p, 0);
  quad_get<F>(P.Z.v, p, 1);
  quad_get<F>(V, p, 2);
  quad_pick<F>(a, P.X.v, H, P.X.v, H);
  mont_mul<F>(p, a, t);      // X H^2, H^3
  quad_get<F>(t, p, 1);
  fe_sub<F>(P.X.v, V, t);
  quad_get<F>(V, p, 0);
  fe_sub<F>(P.X.v, P.X.v, V);
  fe_sub<F>(P.X.v, P.X.v, V);
  fe_sub<F>(V, V, P.X.v);
  quad_pick<F>(a, r, P.Y.v, r, P.Y.v);
  quad_pick<F>(b, V, t, V, t);
  mont_mul<F>(p, a, b);      // r (V - X3), Y H^3
  quad_get<F>(a, p, 0);
  quad_get<F>(b, p, 1);
  fe_sub<F>(P.Y.v, a, b);
}

// ---------------------------------------------------------------- fixed base
// Table of a generator: entry (j, v) = v 2^(16 j) G for v = 1 .. 2^15, j < 16, as
// affine Montgomery points (x limbs, y limbs; row j 2^15 + v - 1).  With signed
// 16-bit digits k G is 16 additions and no doublings (an 8-bit unsigned table
// takes 32).  32 MiB per 256-bit curve (48 MiB for 12 limbs): it stays in the
// 129 MB L2, and a wider window would not.
constexpr int kGWin = 16;
constexpr int kGRows = 16;
constexpr uint32_t kGEntries = 1u << (kGWin - 1);

// a < b for 8-limb integers
ECC_DEV bool lt256(const uint32_t* a, const uint32_t* b) {
  uint32_t t = ptx::sub_cc(a[0], b[0]);
#pragma unroll
  for (int k = 1; k < 8; ++k) t = ptx::subc_cc(a[k], b[k]);
  (void)t;
  return ptx::subc(0, 0) != 0;
}

ECC_DEV bool is_zero256(const uint32_t* a) {
  uint32_t acc = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) acc |= a[k];
  return acc == 0;
}

ECC_DEV void sub256(uint32_t* r, const uint32_t* a, const uint32_t* b) {
  r[0] = ptx::sub_cc(a[0], b[0]);
#pragma unroll
  for (int k = 1; k < 7; ++k) r[k] = ptx::subc_cc(a[k], b[k]);
  r[7] = ptx::subc(a[7], b[7]);
}

// Signed 16-bit digits of k < n: k or n - k, whichever is below 2^255 (its sign
// in `neg`), plus 2^15 in every digit, so that digit j is its 16-bit half minus
// 2^15 without carries.  The ninth word is the last digit's carry.
template <class C>
ECC_DEV void comb_recode(uint32_t* k, bool& neg) {
  uint32_t nn[8], m[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) nn[i] = C::n(i);
  sub256(m, nn, k);
  neg = lt256(m, k);  // n - k < k
#pragma unroll
  for (int i = 0; i < 8; ++i) k[i] = neg ? m[i] : k[i];
  k[0] = ptx::add_cc(k[0], 0x80008000u);
#pragma unroll
  for (int i = 1; i < 8; ++i) k[i] = ptx::addc_cc(k[i], 0x80008000u);
  k[8] = ptx::addc(0, 0);
}

// Digit j of a recoded scalar given its word j >> 1 (in [-2^15, 2^15]).
ECC_DEV int comb_digit(uint32_t word, uint32_t carry, int j) {
  const uint32_t h = (j & 1) ? word >> 16 : word & 0xffffu;
  return (int)h + (j == kGRows - 1 ? (int)(carry << 16) : 0) - 0x8000;
}

// Affine point at row `row` of an AoS array of Montgomery points.
template <class F>
ECC_DEV void load_affine(const uint32_t* base, size_t row, uint32_t* x, uint32_t* y) {
  constexpr int G = F::N / 4;
  const uint4* p = reinterpret_cast<const uint4*>(base) + row * 2 * G;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint4 t = p[g], s = p[G + g];
    x[4 * g] = t.x, x[4 * g + 1] = t.y, x[4 * g + 2] = t.z, x[4 * g + 3] = t.w;
    y[4 * g] = s.x, y[4 * g + 1] = s.y, y[4 * g + 2] = s.z, y[4 * g + 3] = s.w;
  }
}

template <class F>
ECC_DEV void store_affine(uint32_t* base, size_t row, const uint32_t* x, const uint32_t* y) {
  constexpr int G = F::N / 4;
  uint4* p = reinterpret_cast<uint4*>(base) + row * 2 * G;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    p[g] = make_uint4(x[4 * g], x[4 * g + 1], x[4 * g + 2], x[4 * g + 3]);
    p[G + g] = make_uint4(y[4 * g], y[4 * g + 1], y[4 * g + 2], y[4 * g + 3]);
  }
}

// ---------------------------------------------------------------- bytes
ECC_DEV uint32_t bswap32(uint32_t x) { return __byte_perm(x, 0, 0x0123); }

// 8 little-endian limbs from 32 big-endian bytes (word-aligned)
ECC_DEV void load_be256(uint32_t* out, const uint32_t* src) {
#pragma unroll
  for (int k = 0; k < 8; ++k) out[k] = bswap32(src[7 - k]);
}

ECC_DEV void store_be256(uint32_t* dst, const uint32_t* v) {
#pragma unroll
  for (int k = 0; k < 8; ++k) dst[7 - k] = bswap32(v[k]);
}

// Threads of the scalar-multiplication kernels: four CTAs of 128 threads resident
// per SM (128 registers a thread), each CTA's warps in step by a barrier per
// operation so that they share the instructions they fetch.  P-256, one triple /
// 2^20 triples, before the calls: 64 threads without barriers 0.87 / 45.7 ms, 128
// with them 0.88 / 35.0 ms, 256 1.32 / 34.9 ms, 512 2.42 / 34.3 ms.
constexpr int kLadderThreads = 128;
constexpr int kLadderCtasPerSm = 4;

// Items per SM up to which four lanes take one: two CTAs of quads, on which the
// warps' products do not wait for each other yet.  secp256k1 verification by threads /
// quads: 1 triple 0.55 / 0.37 ms, 4096 0.56 / 0.38, 9000 0.57 / 0.52; P-256 0.89 / 0.58,
// 0.89 / 0.58, 0.89 / 0.83.
constexpr size_t kQuadItemsPerSm = 64;

}  // namespace ecc
