// EC-operator launchers: batched affine PADD / PDBL on caller arrays, and the
// per-device generator table v 2^(16 j) G (FPMUL precomputation, Section 2.1.1).
#include <algorithm>
#include <mutex>

#include "internal.h"
#include "ladder.cuh"
#include "ops.cuh"

namespace ecc {

namespace {

template <class C, bool DBL>
cudaError_t point_add(size_t n, const uint32_t* p, const uint32_t* q, uint32_t* out, cudaStream_t st) {
  using F = typename C::Fp;
  constexpr int N = F::N, B = kGasThreads;
  Scratch ws;
  cudaError_t e = point_scratch<F>(ws, n, p, DBL ? nullptr : &q, out, st);
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(GasSmem<N, B>);
  e = cudaFuncSetAttribute(k_point_ops<C, DBL, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_point_ops<C, DBL, B><<<row_ctas(n), B, smem, st>>>(p, q, out, SoA<F>{ws.as<uint4>(), n}, n,
                                                       aligned16(p, DBL ? p : q, out));
  return cudaGetLastError();
}

template <class C>
cudaError_t point_add(size_t n, const uint32_t* p, const uint32_t* q, uint32_t* out, int dbl,
                      cudaStream_t st) {
  return dbl ? point_add<C, true>(n, p, q, out, st) : point_add<C, false>(n, p, q, out, st);
}

// --------------------------------------------------------------- G table

// Entries (j, 1) = 2^(16 j) G of a generator table: one thread's chain of
// doublings, then one lane per row makes its point affine.
template <class C>
__global__ void k_gtable_rows(uint32_t* tab) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  __shared__ uint32_t row[kGRows][3 * N];
  if (threadIdx.x == 0) {
    uint32_t X[N], Y[N], Z[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      X[k] = C::gx(k);
      Y[k] = C::gy(k);
    }
    to_mont<F>(X, X);
    to_mont<F>(Y, Y);
    fe_set_one<F>(Z);
#pragma unroll 1
    for (int s = 0; s < kGWin * kGRows; ++s) {
      if (s % kGWin == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
          row[s / kGWin][k] = X[k];
          row[s / kGWin][N + k] = Y[k];
          row[s / kGWin][2 * N + k] = Z[k];
        }
      }
      jac_dbl_half<C>(X, Y, Z);
    }
  }
  __syncwarp();
  if (threadIdx.x < kGRows) {
    uint32_t X[N], Y[N], Z[N], t[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      X[k] = row[threadIdx.x][k];
      Y[k] = row[threadIdx.x][N + k];
      Z[k] = row[threadIdx.x][2 * N + k];
    }
    fe_inv_mont<F>(Z, Z);
    mont_sqr<F>(t, Z);
    mont_mul<F>(X, X, t);
    mont_mul<F>(t, t, Z);
    mont_mul<F>(Y, Y, t);
    store_affine<F>(tab, (size_t)threadIdx.x * kGEntries, X, Y);
  }
}

// Entries (j, 2^k + u) = (j, 2^k) + (j, u) of every row, u = 1 .. 2^k (the last a
// doubling): a thread does `per` consecutive u with one inversion (Montgomery's
// trick).  All operands are distinct multiples below the group order, so no sum
// is exceptional but the doubling.
constexpr int kGFill = 8;

template <class C>
__global__ void __launch_bounds__(128) k_gtable_fill(uint32_t* tab, int k, int per) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t per_row = (1u << k) / per;
  if (t >= kGRows * per_row) return;
  const size_t base = (size_t)(t / per_row) * kGEntries;
  const uint32_t u0 = 1 + (t % per_row) * per;
  uint32_t xa[N], ya[N], xb[N], yb[N], run[N], d[N], pre[kGFill][N];
  load_affine<F>(tab, base + (1u << k) - 1, xa, ya);
  fe_set_one<F>(run);
  for (int q = 0; q < per; ++q) {
    load_affine<F>(tab, base + u0 + q - 1, xb, yb);
    add_den<C>(d, xa, ya, xb, yb);
    fe_copy<F>(pre[q], run);
    mont_mul<F>(run, run, d);
  }
  fe_inv_mont<F>(run, run);
  for (int q = per - 1; q >= 0; --q) {
    uint32_t inv[N];
    load_affine<F>(tab, base + u0 + q - 1, xb, yb);
    const int kind = add_den<C>(d, xa, ya, xb, yb);
    mont_mul<F>(inv, run, pre[q]);
    mont_mul<F>(run, run, d);
    add_finish<C>(xb, yb, kind, inv, xa, ya, xb, yb);
    store_affine<F>(tab, base + (1u << k) + u0 + q - 1, xb, yb);
  }
}

template <class C>
cudaError_t build_gtable(uint32_t** out, cudaStream_t st) {
  uint32_t* tab = nullptr;
  cudaError_t e = cudaMalloc(&tab, (size_t)kGRows * kGEntries * 2 * C::Fp::N * 4);
  if (e != cudaSuccess) return e;
  k_gtable_rows<C><<<1, 32, 0, st>>>(tab);
  for (int k = 0; k + 1 < kGWin; ++k) {
    const int per = std::min(1 << k, kGFill);
    const unsigned threads = (unsigned)kGRows * ((1u << k) / per);
    k_gtable_fill<C><<<(threads + 127) / 128, 128, 0, st>>>(tab, k, per);
  }
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaFree(tab);
    return e;
  }
  *out = tab;
  return cudaSuccess;
}

std::mutex g_tab_mu;
uint32_t* g_tabs[64][5] = {};

}  // namespace

cudaError_t gtable(int curve, const uint32_t** table, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || curve < 0 || curve > 4) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(g_tab_mu);
  if (!g_tabs[dev][curve]) {
    uint32_t* t = nullptr;
    switch (curve) {
      case 0: e = build_gtable<Secp256k1>(&t, st); break;
      case 1: e = build_gtable<P256>(&t, st); break;
      case 2: e = build_gtable<BN254>(&t, st); break;
      case 3: e = build_gtable<BLS12_381>(&t, st); break;
      case 4: e = build_gtable<SM2>(&t, st); break;
    }
    if (e != cudaSuccess) return e;
    g_tabs[dev][curve] = t;
  }
  *table = g_tabs[dev][curve];
  return cudaSuccess;
}

namespace {

// y^2 = x^3 + a x + b in Montgomery form, canonical coordinates; (0, 0) is O.
template <class C>
__global__ void k_validate(const uint32_t* __restrict__ p, size_t n, uint8_t* __restrict__ ok) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t x[N], y[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    x[k] = p[2 * N * i + k];
    y[k] = p[2 * N * i + N + k];
  }
  if (pt_is_inf<F>(x, y)) {
    ok[i] = 1;
    return;
  }
  if (!fe_lt_modulus<F>(x) || !fe_lt_modulus<F>(y)) {
    ok[i] = 0;
    return;
  }
  to_mont<F>(x, x);
  to_mont<F>(y, y);
  uint32_t lhs[N], rhs[N], t[N];
  mont_sqr<F>(lhs, y);
  mont_sqr<F>(t, x);
  if (!C::A_ZERO) {
    uint32_t a[N];
    curve_a<C>(a);
    fe_add<F>(t, t, a);
  }
  mont_mul<F>(rhs, t, x);
#pragma unroll
  for (int k = 0; k < N; ++k) t[k] = C::b(k);
  fe_add<F>(rhs, rhs, t);
  ok[i] = fe_eq<F>(lhs, rhs) ? 1 : 0;
}

}  // namespace

cudaError_t launch_validate_points(int curve, size_t n, const uint32_t* p, uint8_t* ok, cudaStream_t st) {
  const unsigned b = (unsigned)((n + 255) / 256);
  switch (curve) {
    case 0: k_validate<Secp256k1><<<b, 256, 0, st>>>(p, n, ok); break;
    case 1: k_validate<P256><<<b, 256, 0, st>>>(p, n, ok); break;
    case 2: k_validate<BN254><<<b, 256, 0, st>>>(p, n, ok); break;
    case 3: k_validate<BLS12_381><<<b, 256, 0, st>>>(p, n, ok); break;
    case 4: k_validate<SM2><<<b, 256, 0, st>>>(p, n, ok); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_point_add(int curve, size_t n, const uint32_t* p, const uint32_t* q,
                             uint32_t* out, int dbl, cudaStream_t st) {
  switch (curve) {
    case 0: return point_add<Secp256k1>(n, p, q, out, dbl, st);
    case 1: return point_add<P256>(n, p, q, out, dbl, st);
    case 2: return point_add<BN254>(n, p, q, out, dbl, st);
    case 3: return point_add<BLS12_381>(n, p, q, out, dbl, st);
    case 4: return point_add<SM2>(n, p, q, out, dbl, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ecc
