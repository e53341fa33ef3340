// EC operator layer (Section 3): limb-interleaved SoA storage, the per-CTA
// gather-apply-scatter batch inversion (Section 3.2), and batched affine
// PADD / PDBL rounds with the compress / inverse / DCWPA structure (Section 3.3).
#pragma once
#include <cstddef>
#include <cstdint>

#include "curves_gen.cuh"
#include "fp.cuh"

namespace ecc {

// --------------------------------------------------------------------------
// Column-major ("limb-interleaved") storage of n field elements (Section 3.3,
// cache-efficient data layout): limbs 4g..4g+3 of element i form one 16-byte
// vector at vec[g * stride + i], so a warp reading element i = base + lane of
// one limb group issues 32 consecutive 16-byte loads.
template <class F>
struct SoA {
  static constexpr int G = F::N / 4;
  uint4* vec;
  size_t stride;

  ECC_DEV void load(size_t i, uint32_t* r) const {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      uint4 v = vec[g * stride + i];
      r[4 * g + 0] = v.x;
      r[4 * g + 1] = v.y;
      r[4 * g + 2] = v.z;
      r[4 * g + 3] = v.w;
    }
  }
  ECC_DEV void store(size_t i, const uint32_t* r) const {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      vec[g * stride + i] = make_uint4(r[4 * g + 0], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
    }
  }
};

template <class F>
struct PtSoA {
  SoA<F> x, y;
  ECC_DEV void load(size_t i, uint32_t* px, uint32_t* py) const {
    x.load(i, px);
    y.load(i, py);
  }
  ECC_DEV void store(size_t i, const uint32_t* px, const uint32_t* py) const {
    x.store(i, px);
    y.store(i, py);
  }
};

// Bytes of SoA storage for n elements of field F.
template <class F>
constexpr size_t soa_bytes(size_t n) {
  return n * F::N * 4;
}

// --------------------------------------------------------------------------
// Curve helpers.  Points are affine (x, y) in Montgomery form; the point at
// infinity O is stored as (0, 0), which lies on none of the supported curves
// (b != 0).
template <class C>
ECC_DEV void curve_a(uint32_t* r) {
#pragma unroll
  for (int i = 0; i < C::Fp::N; ++i) r[i] = C::a(i);
}

template <class F>
ECC_DEV bool pt_is_inf(const uint32_t* x, const uint32_t* y) {
  uint32_t acc = 0;
#pragma unroll
  for (int i = 0; i < F::N; ++i) acc |= x[i] | y[i];
  return acc == 0;
}

// 3 x^2 + a (numerator of the PDBL slope, Section 2.1.1)
template <class C>
ECC_DEV void dbl_numerator(uint32_t* num, const uint32_t* x) {
  using F = typename C::Fp;
  uint32_t t[F::N];
  mont_sqr<F>(t, x);
  fe_add<F>(num, t, t);
  fe_add<F>(num, num, t);
  if (!C::A_ZERO) {
    uint32_t a[F::N];
    curve_a<C>(a);
    fe_add<F>(num, num, a);
  }
}

// Classification of P + T for the batched formulas.
enum AddKind : int { ADD_REGULAR = 0, ADD_DOUBLE = 1, ADD_RET_T = 2, ADD_RET_P = 3, ADD_RET_INF = 4 };

// Denominator of lambda for P + T (Eqn 2, or PDBL when P = T), or 1 when the
// result needs no slope (an operand is O, or P = -T).
template <class C>
ECC_DEV int add_kind(const uint32_t* xp, const uint32_t* yp, const uint32_t* xt, const uint32_t* yt) {
  using F = typename C::Fp;
  if (pt_is_inf<F>(xp, yp)) return ADD_RET_T;
  if (pt_is_inf<F>(xt, yt)) return ADD_RET_P;
  if (!fe_eq<F>(xp, xt)) return ADD_REGULAR;
  if (fe_eq<F>(yp, yt) && !fe_is_zero<F>(yp)) return ADD_DOUBLE;
  return ADD_RET_INF;
}

template <class C>
ECC_DEV int add_den(uint32_t* den, const uint32_t* xp, const uint32_t* yp, const uint32_t* xt,
                    const uint32_t* yt) {
  using F = typename C::Fp;
  const int kind = add_kind<C>(xp, yp, xt, yt);
  if (kind == ADD_REGULAR) {
    fe_sub<F>(den, xt, xp);
  } else if (kind == ADD_DOUBLE) {
    fe_add<F>(den, yp, yp);
  } else {
    fe_set_one<F>(den);
  }
  return kind;
}

// Completes R = P + T given kind and inv = 1 / den (Eqn 2-3; PDBL slope for
// ADD_DOUBLE).  R may alias P or T.
template <class C>
ECC_DEV void add_finish(uint32_t* xr, uint32_t* yr, int kind, const uint32_t* inv,
                        const uint32_t* xp, const uint32_t* yp, const uint32_t* xt,
                        const uint32_t* yt) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  if (kind == ADD_REGULAR || kind == ADD_DOUBLE) {
    uint32_t num[N], lam[N], x3[N], t[N];
    if (kind == ADD_REGULAR) {
      fe_sub<F>(num, yt, yp);
    } else {
      dbl_numerator<C>(num, xp);
    }
    mont_mul<F>(lam, num, inv);
    mont_sqr<F>(x3, lam);
    fe_sub<F>(x3, x3, xp);
    fe_sub<F>(x3, x3, xt);
    fe_sub<F>(t, xp, x3);
    mont_mul<F>(t, lam, t);
    fe_sub<F>(yr, t, yp);
    fe_copy<F>(xr, x3);
  } else if (kind == ADD_RET_T) {
    fe_copy<F>(xr, xt);
    fe_copy<F>(yr, yt);
  } else if (kind == ADD_RET_P) {
    fe_copy<F>(xr, xp);
    fe_copy<F>(yr, yp);
  } else {
    fe_set_zero<F>(xr);
    fe_set_zero<F>(yr);
  }
}

// PDBL denominator 2y, or 1 when the result is O (P = O or y = 0).
template <class C>
ECC_DEV bool dbl_den(uint32_t* den, const uint32_t* y) {
  using F = typename C::Fp;
  const bool live = !fe_is_zero<F>(y);
  if (live) {
    fe_add<F>(den, y, y);
  } else {
    fe_set_one<F>(den);
  }
  return live;
}

template <class C>
ECC_DEV void dbl_finish(uint32_t* xr, uint32_t* yr, bool live, const uint32_t* inv,
                        const uint32_t* x, const uint32_t* y) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  if (live) {
    uint32_t num[N], lam[N], x3[N], t[N];
    dbl_numerator<C>(num, x);
    mont_mul<F>(lam, num, inv);
    mont_sqr<F>(x3, lam);
    fe_sub<F>(x3, x3, x);
    fe_sub<F>(x3, x3, x);
    fe_sub<F>(t, x, x3);
    mont_mul<F>(t, lam, t);
    fe_sub<F>(yr, t, y);
    fe_copy<F>(xr, x3);
  } else {
    fe_set_zero<F>(xr);
    fe_set_zero<F>(yr);
  }
}

// --------------------------------------------------------------------------
// Per-CTA gather-apply-scatter inversion (Section 3.2).  Every thread brings
// the product of its own chain; every thread gets back the inverse of its own
// product.  Gather: a butterfly of products over groups of BLOCK / 32 lanes
// (shuffles); apply: the 32 lanes of one warp invert the 32 group products side by
// side (the branch-free divsteps take a full warp no longer than one lane, so the
// groups need no common product); scatter: the butterfly walked back down (each
// level peels the partner subtree).  With 256 threads that is 3 products up and 3
// down instead of 8 and 8 for one inversion of the CTA's whole product: with the
// faster divsteps a BN254 MSM of 4096 points, all of it rounds of this latency,
// takes 3.33 ms instead of 4.48, one of 130003 BLS12-381 points 8.6 instead of 11.0.
// A group is the lanes equal mod 32 / PER, so that its index is a lane's low bits.
// One batch-inversion group per CTA of kGasThreads threads; kGasCtasPerSm such
// CTAs are resident per SM (128 registers per thread), so while one CTA waits
// for its group's inversion the other keeps the SM's multiply-add pipe busy.
// (Measured on GB300: 2 x 256 threads beats 4 x 128, whose halved groups pay
// twice the inversions per item.)
constexpr int kGasThreads = 256;
constexpr int kGasCtasPerSm = 2;
constexpr int kGasResidentThreads = kGasThreads * kGasCtasPerSm;

template <int N, int BLOCK>
struct GasSmem {
  // subtree products per level as 16-byte vectors, thread-fastest (a warp's
  // stores of one vector are 512 contiguous bytes); every thread touches only
  // its own column [.][.][threadIdx.x], which is what lets a kernel reuse the
  // area as per-thread staging outside cta_invert (five elements a thread)
  uint4 tree[5][N / 4][BLOCK];
  uint4 group[N / 4][32];  // group products, then their inverses
};

// The GAS scratch lives in dynamic shared memory (it exceeds the 48 KB static
// limit for 12-limb fields); launches pass sizeof(GasSmem<N, BLOCK>).
template <int N, int BLOCK>
ECC_DEV GasSmem<N, BLOCK>& gas_smem() {
  extern __shared__ __align__(16) unsigned char ecc_dyn_smem[];
  return *reinterpret_cast<GasSmem<N, BLOCK>*>(ecc_dyn_smem);
}

template <class F>
ECC_DEV void fe_shfl_xor(uint32_t* r, const uint32_t* a, int mask) {
#pragma unroll
  for (int i = 0; i < F::N; ++i) r[i] = __shfl_xor_sync(0xffffffffu, a[i], mask);
}

// PLAIN: the inverse as an integer (out = in^-1 mod q up to the tree's factors of
// R) instead of the Montgomery form's in^-1 R^2, for chains over plain integers.
template <class F, int BLOCK, bool PLAIN = false>
__device__ void cta_invert(uint32_t* out, const uint32_t* in, GasSmem<F::N, BLOCK>& sm) {
  constexpr int N = F::N, G = N / 4;
  constexpr int PER = BLOCK / 32;  // lanes of a group
  constexpr int LV = PER <= 1 ? 0 : (PER <= 2 ? 1 : (PER <= 4 ? 2 : (PER <= 8 ? 3 : (PER <= 16 ? 4 : 5))));
  static_assert(BLOCK % 32 == 0 && (1 << LV) == PER, "a power of two warps");
  constexpr unsigned GW = 32 / PER;  // groups of a warp: lanes equal mod GW
  const unsigned tid = threadIdx.x, lane = tid & 31u;
  const unsigned group = (tid >> 5) * GW + (lane & (GW - 1));
  uint32_t v[N], t[N];
  fe_copy<F>(v, in);
#pragma unroll
  for (int l = 0; l < LV; ++l) {
#pragma unroll
    for (int g = 0; g < G; ++g)
      sm.tree[l][g][tid] = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
    fe_shfl_xor<F>(t, v, (int)GW << l);
    mont_mul<F>(v, v, t);
  }
  if (lane < GW) {
#pragma unroll
    for (int g = 0; g < G; ++g)
      sm.group[g][group] = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
  }
  __syncthreads();
  if (tid < 32) {
    uint32_t w[N];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint4 q = sm.group[g][tid];
      w[4 * g] = q.x, w[4 * g + 1] = q.y, w[4 * g + 2] = q.z, w[4 * g + 3] = q.w;
    }
    if constexpr (PLAIN) {
      fe_inv_int<F>(w, w);
    } else {
      fe_inv_mont<F>(w, w);
    }
#pragma unroll
    for (int g = 0; g < G; ++g)
      sm.group[g][tid] = make_uint4(w[4 * g], w[4 * g + 1], w[4 * g + 2], w[4 * g + 3]);
  }
  __syncthreads();
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint4 q = sm.group[g][group];
    v[4 * g] = q.x, v[4 * g + 1] = q.y, v[4 * g + 2] = q.z, v[4 * g + 3] = q.w;
  }
#pragma unroll
  for (int l = LV - 1; l >= 0; --l) {
    uint32_t s[N];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint4 q = sm.tree[l][g][tid];
      s[4 * g] = q.x, s[4 * g + 1] = q.y, s[4 * g + 2] = q.z, s[4 * g + 3] = q.w;
    }
    fe_shfl_xor<F>(t, s, (int)GW << l);
    mont_mul<F>(v, v, t);
  }
  fe_copy<F>(out, v);
  __syncthreads();  // shared storage is reused by the next round
}

// --------------------------------------------------------------------------
// One batched round over the items [begin, end) owned by this CTA (Montgomery's
// trick with the DCWPA step, Section 3.3).  R provides
//   den(i, d)        the denominator of item i,
//   finish(i, inv)   complete item i given inv = 1 / den.
// Compress stores only the running product before each item in M (the
// intermediate array of Section 3.3); DCWPA computes the denominators again.
template <class F, int BLOCK, class R>
__device__ void batch_round(R& rd, size_t begin, size_t end, const SoA<F>& M,
                            GasSmem<F::N, BLOCK>& sm) {
  constexpr int N = F::N;
  uint32_t run[N], d[N];
  fe_set_one<F>(run);
  const size_t i0 = begin + threadIdx.x;
  for (size_t i = i0; i < end; i += BLOCK) {
    M.store(i, run);
    rd.den(i, d);
    mont_mul<F>(run, run, d);
  }
  uint32_t inv[N];
  cta_invert<F, BLOCK>(inv, run, sm);
  if (i0 < end) {
    const size_t last = i0 + ((end - 1 - i0) / BLOCK) * BLOCK;
    for (size_t i = last + BLOCK; i > i0;) {
      i -= BLOCK;
      uint32_t mine[N];
      M.load(i, mine);
      rd.den(i, d);
      mont_mul<F>(mine, inv, mine);
      mont_mul<F>(inv, inv, d);
      rd.finish(i, mine);
    }
  }
}

}  // namespace ecc
