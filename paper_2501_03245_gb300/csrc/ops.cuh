// Kernels on the caller's row-major arrays of canonical limbs: field operations,
// batch inversion (Montgomery's trick with GAS, Section 3.2) and batched point
// addition and doubling (PADD / PDBL, Section 3.3).
//
// The inversion and the point operations compute on the caller's plain integers,
// without converting them: a plain d is the Montgomery form of d R^-1, so a chain
// of Montgomery products of plain values carries a power of R that the inverse of
// the chain's product carries back, and the few results that need the other power
// get it from one product.  One kernel reads each input twice (the second time
// from L2 for arrays up to its size) and writes each output once.
#pragma once
#include <cstddef>
#include <algorithm>
#include <cstdint>

#include "ec.cuh"
#include "internal.h"

namespace ecc {

// ---------------------------------------------------------------- rows

// Rows of N limbs at any 4-byte alignment; `vec`: the array is 16-byte aligned, as
// whole allocations and their rows are, and a row is N / 4 vector accesses.
template <int N>
ECC_DEV void row_load(const uint32_t* base, size_t word, int vec, uint32_t* r) {
  if (vec) {
    const uint4* p = reinterpret_cast<const uint4*>(base + word);
#pragma unroll
    for (int g = 0; g < N / 4; ++g) {
      const uint4 t = p[g];
      r[4 * g] = t.x, r[4 * g + 1] = t.y, r[4 * g + 2] = t.z, r[4 * g + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) r[k] = base[word + k];
  }
}

template <int N>
ECC_DEV void row_store(uint32_t* base, size_t word, int vec, const uint32_t* r) {
  if (vec) {
    uint4* p = reinterpret_cast<uint4*>(base + word);
#pragma unroll
    for (int g = 0; g < N / 4; ++g) p[g] = make_uint4(r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) base[word + k] = r[k];
  }
}

// r mod q for any r < 2^(32 N) (canonical inputs pass the first comparison)
template <class F>
ECC_DEV void fe_canon(uint32_t* r) {
  constexpr int N = F::N;
  if (fe_lt_modulus<F>(r)) return;
  if constexpr (F::FORM == 2) {
    uint32_t t[N + 1];
    fe_copy<F>(t, r);
    t[N] = 0;
    fe_sub_once<F>(r, t);  // 2^256 < 2 q
  } else {
    to_mont<F>(r, r);
    from_mont<F>(r, r);
  }
}

inline int aligned16(const void* a, const void* b, const void* c = nullptr) {
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) &
          15u) == 0;
}

// ---------------------------------------------------------------- unit ops

// out_i = a_i * b_i mod q (a2: Montgomery multiplication, Algorithm 2): one
// factor in Montgomery form makes the product plain.
template <class F>
__global__ void k_fe_mul(const uint32_t* a, const uint32_t* b, uint32_t* out, size_t n, int vec) {
  constexpr int N = F::N;
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t x[N], y[N];
  row_load<N>(a, i * N, vec, x);
  row_load<N>(b, i * N, vec, y);
  to_mont<F>(x, x);
  mont_mul<F>(x, x, y);
  row_store<N>(out, i * N, vec, x);
}

// out_i = a_i + b_i or a_i - b_i mod q (a3)
template <class F>
__global__ void k_fe_addsub(const uint32_t* a, const uint32_t* b, uint32_t* out, size_t n, int subtract,
                            int vec) {
  constexpr int N = F::N;
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t x[N], y[N], z[N];
  row_load<N>(a, i * N, vec, x);
  row_load<N>(b, i * N, vec, y);
  if (subtract) {
    fe_sub<F>(z, x, y);
  } else {
    fe_add<F>(z, x, y);
  }
  row_store<N>(out, i * N, vec, z);
}

// out_i = a_i^-1, 0 -> 0, without scratch: a thread inverts the product of its
// kInvRun elements (a4, a5).  One inversion of a full warp keeps its scheduler
// about a third busy, so four warps a scheduler hide each other.
constexpr int kInvRun = 4;

template <class F>
__global__ void __launch_bounds__(128) k_fe_inv(const uint32_t* a, uint32_t* out, size_t n, int vec) {
  constexpr int N = F::N;
  const size_t T = gridDim.x * (size_t)blockDim.x, t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (size_t i0 = t; i0 < n; i0 += kInvRun * T) {
    uint32_t x[kInvRun][N], pre[kInvRun][N], run[N];
    fe_set_one<F>(run);
#pragma unroll
    for (int k = 0; k < kInvRun; ++k) {
      fe_set_zero<F>(x[k]);
      if (i0 + k * T < n) {
        row_load<N>(a, (i0 + k * T) * N, vec, x[k]);
        fe_canon<F>(x[k]);
      }
      fe_copy<F>(pre[k], run);
      if (!fe_is_zero<F>(x[k])) mont_mul<F>(run, run, x[k]);
    }
    uint32_t in[N], inv[N];
    fe_copy<F>(in, run);
    fe_inv_int<F>(inv, in);
#pragma unroll
    for (int k = kInvRun - 1; k >= 0; --k) {
      if (i0 + k * T >= n) continue;
      uint32_t r[N];
      if (fe_is_zero<F>(x[k])) {
        fe_set_zero<F>(r);
      } else {
        mont_mul<F>(r, inv, pre[k]);
        mont_mul<F>(inv, inv, x[k]);
      }
      row_store<N>(out, (i0 + k * T) * N, vec, r);
    }
  }
}

// ---------------------------------------------------------------- batch inverse

// a5: out_i = a_i^-1, 0 -> 0.  Thread t of the grid's T threads has the elements
// t, t + T, .. (coalesced rows) and their prefix products in M; one inversion per
// eight threads (cta_invert).  The next element's operands are loaded before the
// current one's products.
template <class F, int BLOCK>
__global__ void __launch_bounds__(BLOCK, kGasResidentThreads / BLOCK)
    k_batch_inverse(const uint32_t* a, uint32_t* out, SoA<F> M, size_t n, int vec) {
  constexpr int N = F::N;
  auto& sm = gas_smem<N, BLOCK>();
  const size_t T = gridDim.x * (size_t)BLOCK, t = blockIdx.x * (size_t)BLOCK + threadIdx.x;
  uint32_t run[N], x[N], nx[N], pre[N], npre[N];
  fe_set_one<F>(run);
  if (t < n) row_load<N>(a, t * N, vec, nx);
  for (size_t i = t; i < n; i += T) {
    fe_copy<F>(x, nx);
    if (i + T < n) row_load<N>(a, (i + T) * N, vec, nx);
    fe_canon<F>(x);
    M.store(i, run);
    if (!fe_is_zero<F>(x)) mont_mul<F>(run, run, x);
  }
  uint32_t inv[N];
  cta_invert<F, BLOCK, true>(inv, run, sm);
  if (t >= n) return;
  const size_t last = t + (n - 1 - t) / T * T;
  row_load<N>(a, last * N, vec, nx);
  M.load(last, npre);
  for (size_t i = last;; i -= T) {
    fe_copy<F>(x, nx);
    fe_copy<F>(pre, npre);
    if (i >= T) {  // i = t + k T: another element below
      row_load<N>(a, (i - T) * N, vec, nx);
      M.load(i - T, npre);
    }
    fe_canon<F>(x);
    if (fe_is_zero<F>(x)) {
      fe_set_zero<F>(pre);
    } else {
      mont_mul<F>(pre, inv, pre);
      mont_mul<F>(inv, inv, x);
    }
    row_store<N>(out, i * N, vec, pre);
    if (i < T) break;
  }
}

// ---------------------------------------------------------------- point ops

// (x, y) <- the slope's point: with lr = lambda R, x3 = lambda^2 - xp - xt and
// y3 = lambda (xp - x3) - yp, all plain.
template <class F>
ECC_DEV void plain_finish(uint32_t* x3, uint32_t* y3, const uint32_t* lr, const uint32_t* lam,
                          const uint32_t* xp, const uint32_t* yp, const uint32_t* xt) {
  uint32_t x[F::N], t[F::N];
  mont_mul<F>(x, lr, lam);
  fe_sub<F>(x, x, xp);
  fe_sub<F>(x, x, xt);
  fe_sub<F>(t, xp, x);
  mont_mul<F>(t, lr, t);
  fe_sub<F>(y3, t, yp);
  fe_copy<F>(x3, x);
}

// out_i = p_i + q_i (a6), or 2 p_i with DBL (a7), on plain affine points.  Items
// and prefix products as in k_batch_inverse.  The inverse of a plain denominator
// comes as d^-1 R^2 (cta_invert's Montgomery form), so the slope's product gives
// lambda R, one product with 1 gives lambda, and x3, y3 come out plain.
// The addition's compress step reads y only when an operand may be O or the two x
// agree.
template <class C, bool DBL, int BLOCK>
__device__ void point_ops(const uint32_t* p, const uint32_t* q, uint32_t* out, SoA<typename C::Fp> M,
                          size_t n, int vec) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  auto& sm = gas_smem<N, BLOCK>();
  const size_t T = gridDim.x * (size_t)BLOCK, t = blockIdx.x * (size_t)BLOCK + threadIdx.x;
  auto coord = [&](const uint32_t* base, size_t i, int y, uint32_t* r) {
    row_load<N>(base, i * 2 * N + y * N, vec, r);
    fe_canon<F>(r);
  };
  uint32_t run[N];
  fe_set_one<F>(run);
#pragma unroll 1
  for (size_t i = t; i < n; i += T) {
    uint32_t d[N];
    M.store(i, run);
    if constexpr (DBL) {
      uint32_t y[N];
      coord(p, i, 1, y);
      dbl_den<C>(d, y);
    } else {
      uint32_t x1[N], x2[N];
      coord(p, i, 0, x1);
      coord(q, i, 0, x2);
      if (fe_is_zero<F>(x1) || fe_is_zero<F>(x2) || fe_eq<F>(x1, x2)) {
        uint32_t y1[N], y2[N];
        coord(p, i, 1, y1);
        coord(q, i, 1, y2);
        add_den<C>(d, x1, y1, x2, y2);
      } else {
        fe_sub<F>(d, x2, x1);
      }
    }
    mont_mul<F>(run, run, d);
  }
  uint32_t inv[N];
  cta_invert<F, BLOCK>(inv, run, sm);
  if (t >= n) return;
#pragma unroll 1
  for (size_t i = t + (n - 1 - t) / T * T;; i -= T) {
    uint32_t x1[N], y1[N], x2[N], y2[N], d[N], mine[N];
    M.load(i, mine);
    coord(p, i, 0, x1);
    coord(p, i, 1, y1);
    int kind;
    if constexpr (DBL) {
      fe_copy<F>(x2, x1);
      kind = dbl_den<C>(d, y1) ? ADD_DOUBLE : ADD_RET_INF;
    } else {
      coord(q, i, 0, x2);
      coord(q, i, 1, y2);
      kind = add_den<C>(d, x1, y1, x2, y2);
    }
    mont_mul<F>(mine, inv, mine);  // d^-1 R^2
    mont_mul<F>(inv, inv, d);
    uint32_t lr[N], lam[N];
    if (kind == ADD_REGULAR) {
      if constexpr (!DBL) {
        fe_sub<F>(lr, y2, y1);
        mont_mul<F>(lr, lr, mine);
        from_mont<F>(lam, lr);
      }
    } else if (kind == ADD_DOUBLE) {
      // (3 x^2 + a) R^-1 times d^-1 R^2 is lambda, plain
      uint32_t s[N];
      mont_sqr<F>(s, x1);
      fe_add<F>(lam, s, s);
      fe_add<F>(s, lam, s);
      if (!C::A_ZERO) {
        uint32_t a[N];
        curve_a<C>(a);
        from_mont<F>(a, a);
        from_mont<F>(a, a);
        fe_add<F>(s, s, a);
      }
      mont_mul<F>(lam, s, mine);
      to_mont<F>(lr, lam);
    }
    if (kind == ADD_REGULAR || kind == ADD_DOUBLE) {
      plain_finish<F>(x1, y1, lr, lam, x1, y1, x2);
    } else if (kind == ADD_RET_INF) {
      fe_set_zero<F>(x1);
      fe_set_zero<F>(y1);
    } else if (kind == ADD_RET_T) {
      if constexpr (!DBL) {
        fe_copy<F>(x1, x2);
        fe_copy<F>(y1, y2);
      }
    }
    row_store<N>(out, i * 2 * N, vec, x1);
    row_store<N>(out, i * 2 * N + N, vec, y1);
    if (i < T) break;
  }
}

template <class C, bool DBL, int BLOCK>
__global__ void __launch_bounds__(BLOCK, kGasResidentThreads / BLOCK)
    k_point_ops(const uint32_t* p, const uint32_t* q, uint32_t* out, SoA<typename C::Fp> M, size_t n, int vec) {
  point_ops<C, DBL, BLOCK>(p, q, out, M, n, vec);
}

// CTAs of a grid over n items: up to kGasCtasPerSm resident ones per SM.
inline unsigned row_ctas(size_t n) {
  const size_t ctas = (n + kGasThreads - 1) / kGasThreads;
  return (unsigned)std::min<size_t>(ctas, (size_t)device_sm_count() * kGasCtasPerSm);
}

// Whether out's rows overlap in's without being the same rows: then a row may be
// written before another thread reads it, and the input is copied first.
inline bool shifted_overlap(const void* in, const void* out, size_t bytes) {
  return in != out && overlap(in, bytes, out, bytes);
}

// Scratch of a point operation over n rows: prefix products, then copies of the inputs
// that the output overlaps other than row for row (q null: none).
template <class F>
cudaError_t point_scratch(Scratch& ws, size_t n, const uint32_t*& p, const uint32_t** q, const uint32_t* out,
                          cudaStream_t st) {
  const size_t rows = n * 2 * F::N * 4;
  const bool cp = shifted_overlap(p, out, rows), cq = q && shifted_overlap(*q, out, rows);
  cudaError_t e = ws.alloc(soa_bytes<F>(n) + (cp ? rows : 0) + (cq ? rows : 0), st);
  if (e != cudaSuccess) return e;
  uint32_t* copy = ws.as<uint32_t>() + soa_bytes<F>(n) / 4;
  auto take = [&](const uint32_t*& in) {
    e = cudaMemcpyAsync(copy, in, rows, cudaMemcpyDeviceToDevice, st);
    in = copy;
    copy += rows / 4;
  };
  if (cp) take(p);
  if (cq && e == cudaSuccess) take(*q);
  return e;
}

}  // namespace ecc
