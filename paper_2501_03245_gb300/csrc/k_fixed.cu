// Launchers of batched FPMUL (k G) and batched ECDSA signing.
#include "fixed_base.cuh"
#include "internal.h"

namespace ecc {

namespace {

unsigned ladder_ctas(size_t threads) { return (unsigned)((threads + kLadderThreads - 1) / kLadderThreads); }

// Copies the `rows` inputs of n rows of 32 bytes that are named in `in` into ws and points
// them there.  An item's rows are read by its own thread, while other items' results
// are written already: an output may be an input's buffer row for row, not otherwise.
cudaError_t keep_rows(Scratch& ws, size_t n, const uint32_t** in[], size_t rows, cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
  cudaError_t e = ws.alloc(rows * n * 32, st);
  for (size_t j = 0; j < rows && e == cudaSuccess; ++j) {
    uint32_t* copy = ws.as<uint32_t>() + j * n * 8;
    e = cudaMemcpyAsync(copy, *in[j], n * 32, cudaMemcpyDeviceToDevice, st);
    *in[j] = copy;
  }
  return e;
}

bool use_quads(size_t n) { return n <= (size_t)device_sm_count() * kQuadItemsPerSm; }

template <class C>
cudaError_t fpmul(int curve, size_t n, const uint32_t* k, uint32_t* out, cudaStream_t st) {
  FixedArgs<C> a{};
  cudaError_t e = gtable(curve, &a.TG, st);
  if (e != cudaSuccess) return e;
  a.n = n;
  a.k = k;
  a.out_pt = out;
  Scratch ws;
  const uint32_t** in[] = {&a.k};
  e = keep_rows(ws, n, in, overlap(k, n * 32, out, n * 2 * C::Fp::N * 4) ? 1 : 0, st);
  if (e != cudaSuccess) return e;
  if (use_quads(n)) {
    k_fpmul<C, true><<<ladder_ctas(4 * n), kLadderThreads, 0, st>>>(a);
  } else {
    k_fpmul<C, false><<<ladder_ctas(n), kLadderThreads, 0, st>>>(a);
  }
  return cudaGetLastError();
}

template <class C>
cudaError_t sign(int curve, size_t n, const uint32_t* d, const uint32_t* h, const uint32_t* k, uint32_t* r,
                 uint32_t* s, uint32_t* pub, cudaStream_t st) {
  FixedArgs<C> a{};
  cudaError_t e = gtable(curve, &a.TG, st);
  if (e != cudaSuccess) return e;
  a.n = n;
  a.k = k;
  a.d = d;
  a.e = h;
  a.out_r = r;
  a.out_s = s;
  a.out_pub = pub;
  Scratch ws;
  const uint32_t** in[3];
  size_t rows = 0;
  for (const uint32_t** p : {&a.k, &a.d, &a.e}) {
    auto hit = [&](const uint32_t* out) { return out != *p && overlap(*p, n * 32, out, n * 32); };
    if (hit(r) || hit(s) || overlap(*p, n * 32, pub, n * 64)) in[rows++] = p;
  }
  e = keep_rows(ws, n, in, rows, st);
  if (e != cudaSuccess) return e;
  if (use_quads(n)) {
    k_sign<C, true><<<ladder_ctas(4 * n), kLadderThreads, 0, st>>>(a);
  } else {
    k_sign<C, false><<<ladder_ctas(n), kLadderThreads, 0, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fixed_base_mul(int curve, size_t n, const uint32_t* k, uint32_t* out,
                                  cudaStream_t st) {
  switch (curve) {
    case 0: return fpmul<Secp256k1>(0, n, k, out, st);
    case 1: return fpmul<P256>(1, n, k, out, st);
    case 2: return fpmul<BN254>(2, n, k, out, st);
    case 3: return fpmul<BLS12_381>(3, n, k, out, st);
    case 4: return fpmul<SM2>(4, n, k, out, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_sign(int curve, size_t n, const uint8_t* d, const uint8_t* e, const uint8_t* k,
                        uint8_t* r, uint8_t* s, uint8_t* pub, cudaStream_t st) {
  auto w = [](const uint8_t* p) { return reinterpret_cast<const uint32_t*>(p); };
  auto o = [](uint8_t* p) { return reinterpret_cast<uint32_t*>(p); };
  switch (curve) {
    case 0: return sign<Secp256k1>(0, n, w(d), w(e), w(k), o(r), o(s), o(pub), st);
    case 1: return sign<P256>(1, n, w(d), w(e), w(k), o(r), o(s), o(pub), st);
    case 4: return sign<SM2>(4, n, w(d), w(e), w(k), o(r), o(s), o(pub), st);
  }
  return cudaErrorNotSupported;
}

}  // namespace ecc
