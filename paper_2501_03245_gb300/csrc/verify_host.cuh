// Host launcher of the batched ECDSA verification kernel, included by one
// translation unit per curve so the library builds in parallel.
#pragma once
#include <algorithm>

#include "internal.h"
#include "verify.cuh"

namespace ecc {

namespace verify_detail {

// Items per SM up to which two quads verify one: one CTA.  By one quad / two: 1
// secp256k1 triple 0.367 / 0.318 ms, 4096 (two CTAs per SM) 0.380 / 0.428; P-256 0.576 / 0.547
// and 0.584 / 0.797.
constexpr size_t kPairItemsPerSm = 16;

template <class C>
cudaError_t verify(size_t n, const uint8_t* hash, const uint8_t* r, const uint8_t* s,
                   const uint8_t* pub, uint8_t* ok, cudaStream_t st, int curve) {
  using Fp = typename C::Fp;
  const uint32_t* tg = nullptr;
  cudaError_t e = gtable(curve, &tg, st);
  if (e != cudaSuccess) return e;
  const size_t sms = (size_t)device_sm_count();
  const int lanes = n <= sms * kPairItemsPerSm ? 8 : n <= sms * kQuadItemsPerSm ? 4 : 1;
  const size_t items = kLadderThreads / lanes;
  size_t ctas = (n + items - 1) / items;
  ctas = std::min<size_t>(ctas, (size_t)device_sm_count() * kLadderCtasPerSm);
  // an input that the results overlap is copied: an item's result is written while other
  // items are still to be read
  const uint8_t* in[4] = {hash, r, s, pub};
  const size_t row[4] = {32, 32, 32, 64};
  size_t copies = 0;
  for (int j = 0; j < 4; ++j) copies += overlap(in[j], row[j] * n, ok, n) ? row[j] * n : 0;
  // per slot: table (affine points), H, recoded u1 (9 words) and u2, r: 1640 or 1644 bytes
  constexpr size_t kU2 = QWindows<C>::HALVES * QWindows<C>::WORDS;
  size_t slots, table, h, work;
  Scratch ws;
  for (;; ctas = (ctas + 1) / 2) {  // half the CTAs, with more items each, where it is refused
    slots = ctas * items;
    table = slots * kQTable * 2 * Fp::N * 4;
    h = soa_bytes<Fp>(slots * kQTable);
    work = table + h + (9 + kU2 + 8) * 4 * slots;
    e = ws.alloc(work + copies, st);
    if (e == cudaSuccess) break;
    if (e != cudaErrorMemoryAllocation || ctas == 1) return e;
    cudaGetLastError();
  }
  uint8_t* p = ws.as<uint8_t>();
  uint8_t* copy = p + work;
  for (int j = 0; j < 4; ++j) {
    if (!overlap(in[j], row[j] * n, ok, n)) continue;
    e = cudaMemcpyAsync(copy, in[j], row[j] * n, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    in[j] = copy;
    copy += row[j] * n;
  }
  VerifyArgs<C> a;
  a.n = n;
  a.hash = reinterpret_cast<const uint32_t*>(in[0]);
  a.r = reinterpret_cast<const uint32_t*>(in[1]);
  a.s = reinterpret_cast<const uint32_t*>(in[2]);
  a.pub = reinterpret_cast<const uint32_t*>(in[3]);
  a.ok = ok;
  a.table = reinterpret_cast<uint32_t*>(p);
  a.H = SoA<Fp>{reinterpret_cast<uint4*>(p + table), slots * kQTable};
  a.u1 = reinterpret_cast<uint32_t*>(p + table + h);
  a.u2 = a.u1 + 9 * slots;
  a.rr = a.u2 + kU2 * slots;
  a.TG = tg;
  a.slots = slots;
  if (lanes == 8) {
    k_verify<C, 8><<<(unsigned)ctas, kLadderThreads, 0, st>>>(a);
  } else if (lanes == 4) {
    k_verify<C, 4><<<(unsigned)ctas, kLadderThreads, 0, st>>>(a);
  } else {
    k_verify<C, 1><<<(unsigned)ctas, kLadderThreads, 0, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace verify_detail

}  // namespace ecc
