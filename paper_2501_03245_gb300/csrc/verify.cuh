// Batched ECDSA verification (the ECC algorithm layer over the EC operators).
//
// Verification of (e, r, s, Q) computes R = u1 G + u2 Q with w = s^-1 mod n,
// u1 = e w, u2 = r w, and accepts iff R != O and x_R mod n == r: one fixed-point
// and one unknown-point multiplication (Section 5.2).  One thread does one
// verification from end to end (ladder.cuh):
//
//   * table {Q, 2Q, .., 16Q}: a chain of additions of Q, made affine with one
//     inversion.  An addition leaves Z_k = Z_(k-1) H_k, so 1 / Z_(k-1) is
//     H_k / Z_k and the chain of H replaces Montgomery's prefix products;
//   * u2 Q: signed kQW-bit fixed windows, most significant first: 255 doublings
//     and at most 52 additions of affine table points.  secp256k1 splits u2 = k1 +
//     k2 lambda (glv.cuh): 125 doublings and the same additions, those of k2 with
//     beta x in the place of x (30000 triples 0.89 -> 0.80 ms, one by a thread 0.71 -> 0.55);
//   * u1 G: 16 additions from the generator's table onto the same accumulator
//     (the digits of u1 need no doublings);
//   * x_R mod n == r without an inversion: X = r Z^2 or X = (r + n) Z^2.
//
// The three uses of the addition run through one loop, so its code (about 1900
// instructions) exists once beside the doubling's.  Per thread slot the table (1024
// bytes), the Z ratios (512) and the scalars (104) live in a workspace of 128 MB for a
// full GPU whatever the batch size: with the generator's 32 MiB more than the L2
// holds, and 2^20 triples (0.17 GB of inputs) move 1.5 GB in and 1.5 GB out of DRAM in 33
// ms, which bounds nothing.
#pragma once
#include "glv.cuh"
#include "jac.cuh"

namespace ecc {

template <class C>
struct VerifyArgs {
  using Fp = typename C::Fp;
  size_t n;
  const uint32_t* hash;  // n x 32 bytes big-endian (read as 8 words)
  const uint32_t* r;
  const uint32_t* s;
  const uint32_t* pub;   // n x 64 bytes (x || y) big-endian
  uint8_t* ok;
  uint32_t* table;       // kQTable affine points per slot
  SoA<Fp> H;             // Z ratios of the table's chain, kQTable per slot
  uint32_t* u1;          // recoded u1: word k of a slot at [k * slots + slot], 9 words
  uint32_t* u2;          // recoded u2, likewise: 9 words, or 5 of each half (sign in the top bit)
  uint32_t* rr;          // r, likewise, 8 words
  const uint32_t* TG;    // generator table (ladder.cuh)
  size_t slots;          // threads of the launch
};

// Signed radix-2^kQW digits of a 256-bit scalar.  With 2^(kQW-1) added in every
// digit the digits are the windows minus 2^(kQW-1), in [-16, 15], no carries.
constexpr int kQW = 5;
constexpr int kQTable = 1 << (kQW - 1);

// The windows of u2, or of both halves of a split u2 (word k of half h at row 5 h + k).
template <class C>
struct QWindows {
  static constexpr int HALVES = C::GLV ? 2 : 1;
  static constexpr int BITS = C::GLV ? 128 : 256;
  static constexpr int DIGITS = (BITS + kQW - 1) / kQW;  // of a half
  static constexpr int WORDS = C::GLV ? 5 : 9;
  static constexpr int STEPS = HALVES * DIGITS;
  // the top window has room for u + offset: u < 2^BITS <= 2^(kQW DIGITS - 2)
  static_assert(kQW * DIGITS >= BITS + 2 && kQW * DIGITS < 32 * WORDS, "recoded scalar and sign fit the words");

  // word k of sum_i 2^(kQW - 1) 2^(kQW i), i < DIGITS
  ECC_DEV static constexpr uint32_t offset(int k) {
    uint32_t w = 0;
    for (int i = 0; i < DIGITS; ++i) {
      const int bit = kQW * i + kQW - 1;
      if (bit >> 5 == k) w |= 1u << (bit & 31);
    }
    return w;
  }
};

template <class C>
ECC_DEV bool on_curve_mont(const uint32_t* x, const uint32_t* y) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  uint32_t l[N], rr[N], t[N];
  mont_sqr<F>(l, y);
  mont_sqr<F>(rr, x);
  if (!C::A_ZERO) {
    uint32_t a[N];
    curve_a<C>(a);
    fe_add<F>(rr, rr, a);
  }
  mont_mul<F>(rr, rr, x);
#pragma unroll
  for (int k = 0; k < N; ++k) t[k] = C::b(k);
  fe_add<F>(rr, rr, t);
  return fe_eq<F>(l, rr);
}

// Parses and checks item i (SEC 1 steps 1-3), leaves r, the recoded u1 and u2 and
// the affine Q in the slot and returns whether the item is well-formed; an
// ill-formed one gets stand-ins that keep the arithmetic defined.
template <class C>
ECC_DEV bool verify_prep(const VerifyArgs<C>& a, size_t i, size_t slot) {
  using Fp = typename C::Fp;
  using Fn = typename C::Fn;
  uint32_t r[8], s[8], nn[8], w[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) nn[k] = C::n(k);
  load_be256(r, a.r + 8 * i);
  load_be256(s, a.s + 8 * i);
  bool valid = !is_zero256(r) && !is_zero256(s) && lt256(r, nn) && lt256(s, nn);
  {
    uint32_t qx[8], qy[8], pp[8];
    load_be256(qx, a.pub + 16 * i);
    load_be256(qy, a.pub + 16 * i + 8);
#pragma unroll
    for (int k = 0; k < 8; ++k) pp[k] = Fp::p(k);
    valid = valid && lt256(qx, pp) && lt256(qy, pp) && !(is_zero256(qx) && is_zero256(qy));
    to_mont<Fp>(qx, qx);
    to_mont<Fp>(qy, qy);
    valid = valid && on_curve_mont<C>(qx, qy);
    if (!valid) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        r[k] = s[k] = k == 0 ? 1u : 0u;
        qx[k] = C::gx(k);
        qy[k] = C::gy(k);
      }
      to_mont<Fp>(qx, qx);
      to_mont<Fp>(qy, qy);
    }
    store_affine<Fp>(a.table, slot * kQTable, qx, qy);
  }
  to_mont<Fn>(s, s);
  fe_inv_mont<Fn>(w, s);  // w R
  // one operand in Montgomery form gives the plain product: (w R) r R^-1 = w r
  uint32_t u[9];
#pragma unroll
  for (int k = 0; k < 8; ++k) a.rr[k * a.slots + slot] = r[k];
  mont_mul<Fn>(u, w, r);
  using QWin = QWindows<C>;
  // v + offset in every window, row0 its first row
  auto recode = [&](uint32_t* v, bool neg, int row0) {
    v[0] = ptx::add_cc(v[0], QWin::offset(0));
#pragma unroll
    for (int k = 1; k < QWin::WORDS - 1; ++k) v[k] = ptx::addc_cc(v[k], QWin::offset(k));
    v[QWin::WORDS - 1] = ptx::addc(QWin::offset(QWin::WORDS - 1), 0);
    if (neg) v[QWin::WORDS - 1] |= 0x80000000u;
#pragma unroll
    for (int k = 0; k < QWin::WORDS; ++k) a.u2[(row0 + k) * a.slots + slot] = v[k];
  };
  if constexpr (C::GLV) {
    uint32_t m1[5], m2[5];
    bool n1, n2;
    glv_split<C>(u, m1, n1, m2, n2);
    recode(m1, n1, 0);
    recode(m2, n2, 5);
  } else {
    recode(u, false, 0);
  }
  uint32_t e[8];
  load_be256(e, a.hash + 8 * i);
  if (!lt256(e, nn)) sub256(e, e, nn);  // e < 2^256 < 2n
  mont_mul<Fn>(u, w, e);
  bool neg;
  comb_recode<C>(u, neg);
  u[8] |= neg ? 2u : 0u;
#pragma unroll
  for (int k = 0; k < 9; ++k) a.u1[k * a.slots + slot] = u[k];
  return valid;
}

// The chain's points (X_k, Y_k) and H_k, k = 2 .. kQTable, become affine in
// place; zi = 1 / Z of the last one.
template <class C, bool QUAD>
ECC_DEV void verify_table_affine(const VerifyArgs<C>& a, size_t slot, uint32_t* zi) {
  using F = typename C::Fp;
  constexpr int N = F::N;
#pragma unroll 1
  for (int k = kQTable; k >= 2; --k) {
    uint32_t x[N], y[N], t[N], h[N];
    const size_t row = slot * kQTable + k - 1;
    load_affine<F>(a.table, row, x, y);
    a.H.load((size_t)(k - 1) * a.slots + slot, h);
    if constexpr (QUAD) {
      __syncwarp();  // every lane of the item has its operands before one stores the row
      uint32_t u[N], p[N];
      quad_pick<F>(u, zi, h, zi, h);
      mont_mul<F>(p, u, zi);  // zi^2, zi h
      quad_get<F>(t, p, 0);
      quad_pick<F>(u, x, zi, x, zi);
      quad_get<F>(zi, p, 1);
      mont_mul<F>(p, u, t);   // x zi^2, zi^3
      quad_get<F>(x, p, 0);
      quad_get<F>(t, p, 1);
      mont_mul<F>(y, y, t);
    } else {
      call_sqr<F>(t, zi);
      call_mul<F>(x, x, t);
      call_mul<F>(t, t, zi);
      call_mul<F>(y, y, t);
      call_mul<F>(zi, zi, h);
    }
    store_affine<F>(a.table, row, x, y);
  }
}

// LANES = 4: four lanes per item, each doing all of it but the products of the group
// operations, which they share; what they store they store alike.  LANES = 8: two
// such quads per item, which sum one part of u1 G + u2 Q each (the halves of a split
// u2 and of u1's rows, or u2 Q and u1 G) and add the two at the end.
template <class C, int LANES>
__global__ void __launch_bounds__(kLadderThreads, LANES > 1 ? 2 : kLadderCtasPerSm) k_verify(VerifyArgs<C> a) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  static_assert(N == 8 && C::Fn::N == 8, "256-bit curves");
  using QWin = QWindows<C>;
  constexpr bool QUAD = LANES > 1, PAIR = LANES == 8;
  constexpr int kSteps = PAIR ? QWin::DIGITS : QWin::STEPS;          // additions of table points
  constexpr int kRows = !PAIR ? kGRows : C::GLV ? kGRows / 2 : 0;  // further additions of G's
  const bool second = PAIR && (threadIdx.x & 4u);                  // the item's second quad
  constexpr int kItems = kLadderThreads / LANES;  // of a CTA
  const size_t own = threadIdx.x / LANES;
  const size_t slot = blockIdx.x * (size_t)kItems + own;
  // threads past the batch repeat its last item (the barriers need every thread)
#pragma unroll 1
  for (size_t i0 = blockIdx.x * (size_t)kItems; i0 < a.n; i0 += a.slots) {
    const bool mine = i0 + own < a.n;
    const size_t i = mine ? i0 + own : a.n - 1;
    const bool valid = verify_prep<C>(a, i, slot);
    JacReg<F> P;
    uint32_t* const X = P.X.v;
    uint32_t* const Y = P.Y.v;
    uint32_t* const Z = P.Z.v;
    uint32_t H[N], x[N], y[N];
    auto dbl = [&]() {
      if constexpr (QUAD) {
        quad_dbl<C>(P);
      } else {
        jac_dbl_half<C>(X, Y, Z);
      }
    };
    // table chain: 2Q by doubling (Z = y_Q), then + Q up to kQTable Q
    load_affine<F>(a.table, slot * kQTable, X, Y);
    fe_set_one<F>(Z);
    dbl();
    a.H.store(a.slots + slot, Z);
    store_affine<F>(a.table, slot * kQTable + 1, X, Y);
    constexpr int kChain = kQTable - 2;
#pragma unroll 1
    for (int it = 0; it < kChain + kSteps + kRows; ++it) {
      int d;
      const uint32_t* src;
      size_t row;
      bool phi = false;  // the point's image under the endomorphism
      auto g_row = [&](int j) {
        const uint32_t c = a.u1[8 * a.slots + slot];
        d = comb_digit(a.u1[(j >> 1) * a.slots + slot], c & 1u, j);
        src = a.TG;
        row = (size_t)j * kGEntries + (d < 0 ? -d : d) - 1;
        if (c & 2u) d = -d;
      };
      if (it < kChain) {
        d = 1;
        src = a.table;
        row = slot * kQTable;
      } else if (it < kChain + kSteps) {
        const int step = it - kChain;
        // the quads of a pair have a half of a split scalar each, else they take turns
        const int half = !C::GLV ? 0 : PAIR ? (int)second : step & 1;
        const int w = QWin::DIGITS - 1 - (PAIR ? step : step / QWin::HALVES);
        const bool only_g = PAIR && !C::GLV && second;
        if (step == 0) {
          fe_inv_mont<F>(x, Z);
          verify_table_affine<C, QUAD>(a, slot, x);
          fe_set_zero<F>(Z);
        } else if (PAIR || half == 0) {
#pragma unroll 1
          for (int k = 0; k < kQW; ++k) {
            __syncthreads();
            if (!only_g) dbl();
          }
        }
        if (only_g) {
          d = 0;
          src = a.TG;
          row = 0;
          if (step < kGRows) g_row(step);
        } else {
          const int bit = kQW * w, wd = bit >> 5, sh = bit & 31;
          const uint32_t* u2 = a.u2 + 5 * half * a.slots + slot;
          uint32_t v = u2[wd * a.slots] >> sh;
          if (sh > 32 - kQW) v |= u2[(wd + 1) * a.slots] << (32 - sh);
          d = (int)(v & (2 * kQTable - 1)) - kQTable;
          src = a.table;
          row = slot * kQTable + (d < 0 ? -d : d) - 1;
          if constexpr (C::GLV) {
            if (u2[4 * a.slots] >> 31) d = -d;
            phi = half != 0;
          }
        }
      } else {
        g_row(it - kChain - kSteps + (second ? kRows : 0));
      }
      __syncthreads();
      if (d != 0) {
        load_affine<F>(src, row, x, y);
        if (d < 0) fe_neg<F>(y, y);
        if constexpr (C::GLV) {
          if (phi) {
            uint32_t beta[N];
#pragma unroll
            for (int k = 0; k < N; ++k) beta[k] = C::glv_beta(k);
            call_mul<F>(x, x, beta);
          }
        }
        if constexpr (QUAD) {
          quad_madd<C>(P, x, y, H);
        } else {
          jac_madd<C>(X, Y, Z, x, y, H);
        }
      }
      if (it < kChain) {
        a.H.store((size_t)(it + 2) * a.slots + slot, H);
        store_affine<F>(a.table, slot * kQTable + it + 2, X, Y);
      }
    }
    if constexpr (PAIR) {  // the other quad's part
      __syncwarp();
      JacReg<F> Q;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        Q.X.v[k] = __shfl_xor_sync(0xffffffffu, X[k], 4);
        Q.Y.v[k] = __shfl_xor_sync(0xffffffffu, Y[k], 4);
        Q.Z.v[k] = __shfl_xor_sync(0xffffffffu, Z[k], 4);
      }
      quad_add<C>(P, Q);
    }
    // R != O and x_R mod n == r, i.e. X = r Z^2 or (r + n < p) X = (r + n) Z^2
    uint32_t r[8], t[8], zz[8], pp[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) r[k] = a.rr[k * a.slots + slot];
    mont_sqr<F>(zz, Z);
    to_mont<F>(t, r);
    mont_mul<F>(t, t, zz);
    bool ok = fe_eq<F>(t, X);
    r[0] = ptx::add_cc(r[0], C::n(0));
#pragma unroll
    for (int k = 1; k < 8; ++k) r[k] = ptx::addc_cc(r[k], C::n(k));
    const bool over = ptx::addc(0, 0) != 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) pp[k] = F::p(k);
    if (!ok && !over && lt256(r, pp)) {
      to_mont<F>(t, r);
      mont_mul<F>(t, t, zz);
      ok = fe_eq<F>(t, X);
    }
    ok = ok && valid && !fe_is_zero<F>(Z);
    if (mine) a.ok[i] = ok ? 1 : 0;
    if constexpr (QUAD) __syncwarp();  // the slot is free
  }
}

}  // namespace ecc
