// Jacobian-coordinate point arithmetic (x = X/Z^2, y = Y/Z^3, Z = 0 for O; Section
// 2.1.2, Table 1) of the MSM, on curves with a = 0: sums that no other thread waits
// for (jac_addto, by one thread, products called as in ladder.cuh) and the short
// dependent chains at the end of a call (quad_*, four lanes a point).
//
// A chain of group operations by one thread costs a product's latency for each of
// an operation's products (16 for an addition, 7 for a doubling; 0.42 us each with
// 8 limbs, 0.9 with 12); a quad (ladder.cuh) takes 5 steps and 3.
#pragma once
#include "ladder.cuh"

namespace ecc {

template <class F>
struct Jac {
  uint32_t X[F::N], Y[F::N], Z[F::N];
};

template <class F>
ECC_DEV void jac_load(const Jac<F>* p, uint32_t* X, uint32_t* Y, uint32_t* Z) {
  constexpr int G = F::N / 4;
  const uint4* v = reinterpret_cast<const uint4*>(p);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint4 a = v[g], b = v[G + g], c = v[2 * G + g];
    X[4 * g] = a.x, X[4 * g + 1] = a.y, X[4 * g + 2] = a.z, X[4 * g + 3] = a.w;
    Y[4 * g] = b.x, Y[4 * g + 1] = b.y, Y[4 * g + 2] = b.z, Y[4 * g + 3] = b.w;
    Z[4 * g] = c.x, Z[4 * g + 1] = c.y, Z[4 * g + 2] = c.z, Z[4 * g + 3] = c.w;
  }
}

template <class F>
ECC_DEV void jac_store(Jac<F>* p, const uint32_t* X, const uint32_t* Y, const uint32_t* Z) {
  constexpr int G = F::N / 4;
  uint4* v = reinterpret_cast<uint4*>(p);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    v[g] = make_uint4(X[4 * g], X[4 * g + 1], X[4 * g + 2], X[4 * g + 3]);
    v[G + g] = make_uint4(Y[4 * g], Y[4 * g + 1], Y[4 * g + 2], Y[4 * g + 3]);
    v[2 * G + g] = make_uint4(Z[4 * g], Z[4 * g + 1], Z[4 * g + 2], Z[4 * g + 3]);
  }
}

template <class F>
ECC_DEV void jac_set_inf(uint32_t* X, uint32_t* Y, uint32_t* Z) {
  fe_set_one<F>(X);
  fe_set_one<F>(Y);
  fe_set_zero<F>(Z);
}

// P <- P + Q, every case of the group law (12 products and 4 squares).
template <class C>
ECC_DEV void jac_addto(uint32_t* X1, uint32_t* Y1, uint32_t* Z1, const uint32_t* X2, const uint32_t* Y2,
                       const uint32_t* Z2) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  if (fe_is_zero<F>(Z2)) return;
  if (fe_is_zero<F>(Z1)) {
    fe_copy<F>(X1, X2);
    fe_copy<F>(Y1, Y2);
    fe_copy<F>(Z1, Z2);
    return;
  }
  uint32_t a[N], H[N], r[N], U[N], S[N];
  call_sqr<F>(a, Z2);
  call_mul<F>(U, X1, a);   // U1
  call_mul<F>(a, a, Z2);
  call_mul<F>(S, Y1, a);   // S1
  call_sqr<F>(a, Z1);
  call_mul<F>(H, X2, a);
  fe_sub<F>(H, H, U);      // U2 - U1
  call_mul<F>(a, a, Z1);
  call_mul<F>(r, Y2, a);
  fe_sub<F>(r, r, S);      // S2 - S1
  if (fe_is_zero<F>(H)) {
    if (fe_is_zero<F>(r)) {
      jac_dbl_rare<C>(X1, Y1, Z1);
    } else {
      jac_set_inf<F>(X1, Y1, Z1);
    }
    return;
  }
  call_mul<F>(Z1, Z1, Z2);
  call_mul<F>(Z1, Z1, H);
  call_sqr<F>(a, H);
  call_mul<F>(U, U, a);    // V = U1 H^2
  call_mul<F>(H, H, a);    // H^3
  call_sqr<F>(X1, r);
  fe_sub<F>(X1, X1, H);
  fe_sub<F>(X1, X1, U);
  fe_sub<F>(X1, X1, U);
  fe_sub<F>(U, U, X1);
  call_mul_sub<F>(Y1, r, U, S, H);
}

// P <- P + Q by a quad, every case of the group law
template <class C>
ECC_DEV void quad_add(JacReg<typename C::Fp>& P, JacReg<typename C::Fp> Q) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  if (fe_is_zero<F>(Q.Z.v)) return;
  if (fe_is_zero<F>(P.Z.v)) {
    P = Q;
    return;
  }
  uint32_t a[N], b[N], p[N], ZZ[N], H[N], r[N];
  quad_pick<F>(a, P.Z.v, Q.Z.v, P.Z.v, P.Z.v);
  quad_pick<F>(b, P.Z.v, Q.Z.v, Q.Z.v, Q.Z.v);
  mont_mul<F>(p, a, b);    // Z1^2, Z2^2, Z1 Z2
  quad_get<F>(ZZ, p, 2);
  quad_get<F>(H, p, 0);    // Z1^2
  quad_get<F>(r, p, 1);    // Z2^2
  quad_pick<F>(a, P.X.v, Q.X.v, Q.Z.v, P.Z.v);
  quad_pick<F>(b, r, H, r, H);
  mont_mul<F>(p, a, b);    // U1, U2, Z2^3, Z1^3
  quad_get<F>(P.X.v, p, 0);
  quad_get<F>(H, p, 1);
  fe_sub<F>(H, H, P.X.v);
  quad_get<F>(Q.Z.v, p, 2);
  quad_get<F>(P.Z.v, p, 3);
  quad_pick<F>(a, P.Y.v, Q.Y.v, H, ZZ);
  quad_pick<F>(b, Q.Z.v, P.Z.v, H, H);
  mont_mul<F>(p, a, b);    // S1, S2, H^2, Z3
  quad_get<F>(Q.X.v, p, 0);
  quad_get<F>(r, p, 1);
  fe_sub<F>(r, r, Q.X.v);
  if (fe_is_zero<F>(H)) {
    // equal points: the doubling of (U1, S1, Z1 Z2), which is the same point
    fe_copy<F>(P.Y.v, Q.X.v);
    fe_copy<F>(P.Z.v, ZZ);
    if (fe_is_zero<F>(r)) {
      jac_dbl_rare<C>(P.X.v, P.Y.v, P.Z.v);
    } else {
      jac_set_inf<F>(P.X.v, P.Y.v, P.Z.v);
    }
    return;
  }
  quad_get<F>(ZZ, p, 2);
  quad_get<F>(P.Z.v, p, 3);
  quad_pick<F>(a, H, P.X.v, r, r);
  quad_pick<F>(b, ZZ, ZZ, r, r);
  mont_mul<F>(p, a, b);    // H^3, V = U1 H^2, r^2
  quad_get<F>(H, p, 0);
  quad_get<F>(ZZ, p, 1);
  quad_get<F>(P.X.v, p, 2);
  fe_sub<F>(P.X.v, P.X.v, H);
  fe_sub<F>(P.X.v, P.X.v, ZZ);
  fe_sub<F>(P.X.v, P.X.v, ZZ);
  fe_sub<F>(ZZ, ZZ, P.X.v);
  quad_pick<F>(a, r, Q.X.v, r, r);
  quad_pick<F>(b, ZZ, H, ZZ, ZZ);
  mont_mul<F>(p, a, b);    // r (V - X3), S1 H^3
  quad_get<F>(a, p, 0);
  quad_get<F>(b, p, 1);
  fe_sub<F>(P.Y.v, a, b);
}

template <class F>
ECC_DEV JacReg<F> quad_load(const Jac<F>* p) {
  JacReg<F> P;
  jac_load<F>(p, P.X.v, P.Y.v, P.Z.v);
  return P;
}

// Jacobian -> affine (x, y) in Montgomery form, (0, 0) for O (one inversion).
template <class F>
ECC_DEV void jac_to_affine(uint32_t* x, uint32_t* y, const JacReg<F>& P) {
  uint32_t zi[F::N], t[F::N];
  fe_inv_mont<F>(zi, P.Z.v);  // 0 for O
  mont_sqr<F>(t, zi);
  mont_mul<F>(x, P.X.v, t);
  mont_mul<F>(t, t, zi);
  mont_mul<F>(y, P.Y.v, t);
}

}  // namespace ecc
