// Batched fixed-point multiplication (FPMUL, Section 2.1.1 / Table 5) and
// batched ECDSA signing (Section 5.2: one modinv plus one FPMUL), one thread per
// item (ladder.cuh): k G is 16 additions of entries of the generator's table,
// then one inversion makes the result affine.  A signature does k G and d G one
// after the other through the same loop and inverts both Z together.  Small batches
// (QUAD) take the four lanes of a quad per item, which do all of it alike but the
// products of the additions.
#pragma once
#include "ladder.cuh"

namespace ecc {

template <class C>
struct FixedArgs {
  size_t n;
  const uint32_t* k;        // FPMUL: n x 8 LE limbs; signing: n x 32 BE bytes (nonce)
  const uint32_t* d;        // signing: private keys, 32 BE bytes
  const uint32_t* e;        // signing: hashes, 32 BE bytes
  uint32_t* out_pt;         // FPMUL: n x 2N LE limbs (affine, (0,0) = O)
  uint32_t* out_r;          // signing: n x 32 BE bytes
  uint32_t* out_s;          // signing: n x 32 BE bytes
  uint32_t* out_pub;        // signing: n x 64 BE bytes
  const uint32_t* TG;       // generator table (ladder.cuh)
};

// k mod n for any 256-bit k (n > 2^253: at most a few subtractions)
template <class C>
ECC_DEV void scalar_mod_n(uint32_t* k) {
  uint32_t nn[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) nn[q] = C::n(q);
#pragma unroll 1
  while (!lt256(k, nn)) sub256(k, k, nn);
}

// P += digit j of the recoded scalar kr (9 words) times 2^(16 j) G
template <class C, bool QUAD>
ECC_DEV void comb_add(const uint32_t* TG, uint32_t word, uint32_t carry, bool neg, int j,
                      JacReg<typename C::Fp>& P) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const int d = comb_digit(word, carry, j);
  if (d == 0) return;
  uint32_t x[N], y[N], H[N];
  load_affine<F>(TG, (size_t)j * kGEntries + (d < 0 ? -d : d) - 1, x, y);
  if ((d < 0) != neg) fe_neg<F>(y, y);
  if constexpr (QUAD) {
    quad_madd<C>(P, x, y, H);
  } else {
    jac_madd<C>(P.X.v, P.Y.v, P.Z.v, x, y, H);
  }
}

// This thread's item: its number and whether it writes the results.  Threads past the
// batch repeat its last item (the barriers need every thread).
template <bool QUAD>
ECC_DEV size_t comb_item(size_t n, bool& writes) {
  const size_t t = blockIdx.x * (size_t)kLadderThreads + threadIdx.x, g = QUAD ? t / 4 : t;
  writes = g < n && (!QUAD || (t & 3) == 0);
  return g < n ? g : n - 1;
}

template <class C, bool QUAD>
__global__ void __launch_bounds__(kLadderThreads, QUAD ? 2 : kLadderCtasPerSm) k_fpmul(FixedArgs<C> a) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  bool writes;
  const size_t i = comb_item<QUAD>(a.n, writes);
  uint32_t k[9];
#pragma unroll
  for (int q = 0; q < 8; ++q) k[q] = a.k[8 * i + q];
  scalar_mod_n<C>(k);
  bool neg;
  comb_recode<C>(k, neg);
  JacReg<F> P;
  uint32_t* const X = P.X.v;
  uint32_t* const Y = P.Y.v;
  uint32_t* const Z = P.Z.v;
  fe_set_zero<F>(X);
  fe_set_zero<F>(Y);
  fe_set_zero<F>(Z);
#pragma unroll 1
  for (int j = 0; j < kGRows; ++j) {
    __syncthreads();
    comb_add<C, QUAD>(a.TG, k[0], k[8], neg, j, P);
    if (j & 1) {  // next word
#pragma unroll
      for (int q = 0; q < 7; ++q) k[q] = k[q + 1];
    }
  }
  uint32_t zi[N], t[N];
  fe_inv_mont<F>(zi, Z);  // 0 for O, which gives (0, 0)
  mont_sqr<F>(t, zi);
  mont_mul<F>(X, X, t);
  mont_mul<F>(t, t, zi);
  mont_mul<F>(Y, Y, t);
  from_mont<F>(X, X);
  from_mont<F>(Y, Y);
  if constexpr (QUAD) __syncwarp();  // the scalar may be in the output's buffer
  if (!writes) return;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    a.out_pt[2 * N * i + q] = X[q];
    a.out_pt[2 * N * i + N + q] = Y[q];
  }
}

// r = x(k G) mod n, s = k^-1 (e + r d) mod n and the public key d G.
template <class C, bool QUAD>
__global__ void __launch_bounds__(kLadderThreads, QUAD ? 2 : kLadderCtasPerSm) k_sign(FixedArgs<C> a) {
  using F = typename C::Fp;
  using Fn = typename C::Fn;
  constexpr int N = F::N;
  static_assert(N == 8 && Fn::N == 8, "256-bit curves");
  bool writes;
  const size_t i = comb_item<QUAD>(a.n, writes);
  uint32_t nn[8], kr[9];
#pragma unroll
  for (int q = 0; q < 8; ++q) nn[q] = C::n(q);
  bool valid;
  {
    uint32_t k[8], d[8];
    load_be256(k, a.k + 8 * i);
    load_be256(d, a.d + 8 * i);
    valid = !is_zero256(k) && !is_zero256(d) && lt256(k, nn) && lt256(d, nn);
  }
  // an ill-formed item signs with k = d = 1; its r and s are discarded
  auto scalar = [&](const uint32_t* src, uint32_t* v) {
    load_be256(v, src + 8 * i);
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = valid ? v[q] : (q == 0 ? 1u : 0u);
  };
  JacReg<F> P;
  uint32_t* const X = P.X.v;
  uint32_t* const Y = P.Y.v;
  uint32_t* const Z = P.Z.v;
  uint32_t Kx[N], Kz[N];
  bool neg = false;
#pragma unroll 1
  for (int j = 0; j < 2 * kGRows; ++j) {  // k G, then d G
    if ((j & (kGRows - 1)) == 0) {
      if (j) {
        fe_copy<F>(Kx, X);  // r needs only x
        fe_copy<F>(Kz, Z);
      }
      scalar(j ? a.d : a.k, kr);
      comb_recode<C>(kr, neg);
      fe_set_zero<F>(Z);
    }
    __syncthreads();
    comb_add<C, QUAD>(a.TG, kr[0], kr[8], neg, j & (kGRows - 1), P);
    if (j & 1) {
#pragma unroll
      for (int q = 0; q < 7; ++q) kr[q] = kr[q + 1];
    }
  }
  // 0 < k, d < n: neither result is O.  1 / Z and 1 / Kz from one inversion
  uint32_t zi[N], t[N];
  mont_mul<F>(t, Z, Kz);
  fe_inv_mont<F>(t, t);
  mont_mul<F>(zi, t, Kz);
  mont_mul<F>(Kz, t, Z);
  mont_sqr<F>(t, zi);
  mont_mul<F>(X, X, t);
  mont_mul<F>(t, t, zi);
  mont_mul<F>(Y, Y, t);
  from_mont<F>(X, X);
  from_mont<F>(Y, Y);
  mont_sqr<F>(t, Kz);
  mont_mul<F>(Kx, Kx, t);
  uint32_t r[8], s[8], v[8], w[8];
  from_mont<F>(r, Kx);
  if (!lt256(r, nn)) sub256(r, r, nn);  // x < p < 2n
  scalar(a.d, v);
  to_mont<Fn>(v, v);
  mont_mul<Fn>(s, v, r);  // d r
  load_be256(w, a.e + 8 * i);
  if (!lt256(w, nn)) sub256(w, w, nn);
  fe_add<Fn>(s, s, w);
  scalar(a.k, v);
  to_mont<Fn>(v, v);
  fe_inv_mont<Fn>(v, v);
  mont_mul<Fn>(s, v, s);  // (k^-1 R) (e + r d) R^-1
  const bool good = valid && !is_zero256(r) && !is_zero256(s);
  if (!good) {
    fe_set_zero<Fn>(r);
    fe_set_zero<Fn>(s);
  }
  // every input of this item has been read: an output may be an input's buffer
  if constexpr (QUAD) __syncwarp();
  if (!writes) return;
  store_be256(a.out_r + 8 * i, r);
  store_be256(a.out_s + 8 * i, s);
  store_be256(a.out_pub + 16 * i, X);
  store_be256(a.out_pub + 16 * i + 8, Y);
}

}  // namespace ecc
