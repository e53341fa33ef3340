"""The reduction tree's kernel (k_msm_tree) run on the host, a thread for each of the
CTA's, where the first lane of every quad runs ahead of the other three as far as the
kernel's own barriers and exchanges let it.  CUDA promises no more than those, so a
lane must not overwrite what the others of its quad have still to read."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import curves, ec
from paper_2501_03245_gb300 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_03245_gb300", "csrc")

PTX = """
#pragma once
#include <cstdint>
namespace ptx {
inline thread_local uint32_t cc = 0;
inline uint32_t put(uint64_t v) { cc = (uint32_t)(v >> 32) != 0; return (uint32_t)v; }
inline uint32_t add_cc(uint32_t a, uint32_t b) { return put((uint64_t)a + b); }
inline uint32_t addc_cc(uint32_t a, uint32_t b) { return put((uint64_t)a + b + cc); }
inline uint32_t addc(uint32_t a, uint32_t b) { return a + b + cc; }
inline uint32_t sub_cc(uint32_t a, uint32_t b) { return put((uint64_t)a - b); }
inline uint32_t subc_cc(uint32_t a, uint32_t b) { return put((uint64_t)a - b - cc); }
inline uint32_t subc(uint32_t a, uint32_t b) { return a - b - cc; }
inline uint32_t lo(uint32_t a, uint32_t b) { return a * b; }
inline uint32_t hi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
inline uint32_t mad_lo_cc(uint32_t a, uint32_t b, uint32_t c) { return put((uint64_t)lo(a, b) + c); }
inline uint32_t madc_lo_cc(uint32_t a, uint32_t b, uint32_t c) { return put((uint64_t)lo(a, b) + c + cc); }
inline uint32_t mad_hi_cc(uint32_t a, uint32_t b, uint32_t c) { return put((uint64_t)hi(a, b) + c); }
inline uint32_t madc_hi_cc(uint32_t a, uint32_t b, uint32_t c) { return put((uint64_t)hi(a, b) + c + cc); }
inline uint32_t madc_hi(uint32_t a, uint32_t b, uint32_t c) { return hi(a, b) + c + cc; }
inline void cp_async16(void*, const void*) {}
inline void cp_async_commit() {}
inline void cp_async_wait_all() {}
inline void cp_async_wait_prior() {}
}
"""

# Threads of one CTA under a lock: a thread runs until it waits for others (a barrier or
# an exchange, named by its members) or ends; the lowest waiting-to-run lane of a quad,
# then the lowest thread, goes next.  Members that have all arrived go on; if none can
# run and some still wait, their partners are gone: the run is stuck.
SRC = """
#define ECC_DEV inline
#define __device__
#define __host__
#define __global__
#define __shared__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __align__(x)
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>
struct alignas(16) uint4 { uint32_t x, y, z, w; };
inline uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }
struct Dim { unsigned x = 1, y = 1, z = 1; };
inline thread_local Dim threadIdx, blockIdx;
inline Dim blockDim, gridDim;
inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, int s) {
  return (uint32_t)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32);
}
inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, int s) {
  return (uint32_t)((((uint64_t)hi << 32) | lo) >> (s & 31));
}
inline uint32_t __byte_perm(uint32_t x, uint32_t, uint32_t) { return __builtin_bswap32(x); }

struct Stuck {};
constexpr int T = 128;
enum State { READY, WAIT, DONE };
struct Cta {
  std::mutex mu;
  std::condition_variable cv;
  State state[T];
  uint32_t word[T];
  std::vector<int> with[T];  // whom a waiting thread waits for
  int run = -1;
  bool stuck = false;
  void next() {  // hands the CTA to the next thread
    for (int t = 0; t < T; ++t) {
      if (state[t] != WAIT) continue;
      bool all = true;
      for (int o : with[t]) all &= state[o] == WAIT && with[o] == with[t];
      if (all) {
        const std::vector<int> go = with[t];
        for (int o : go) state[o] = READY;
      }
    }
    int best = -1;
    for (int lane = 0; lane < 4 && best < 0; ++lane)
      for (int t = lane; t < T && best < 0; t += 4)
        if (state[t] == READY) best = t;
    run = best;
    if (best < 0)
      for (int t = 0; t < T; ++t) stuck |= state[t] == WAIT;
    cv.notify_all();
  }
  void wait_turn(std::unique_lock<std::mutex>& l, int t) {
    cv.wait(l, [&] { return run == t || stuck; });
    if (stuck) throw Stuck{};
  }
  void meet(const std::vector<int>& members) {
    const int t = (int)threadIdx.x;
    std::unique_lock<std::mutex> l(mu);
    with[t] = members;
    state[t] = WAIT;
    next();
    wait_turn(l, t);
  }
} cta;

inline std::vector<int> lanes(unsigned mask) {
  std::vector<int> v;
  for (int i = 0; i < 32; ++i)
    if (mask >> i & 1u) v.push_back((int)(threadIdx.x & ~31u) + i);
  return v;
}
inline void __syncwarp(unsigned mask = 0xffffffffu) { cta.meet(lanes(mask)); }
inline void __syncthreads() {
  std::vector<int> v;
  for (int t = 0; t < T; ++t) v.push_back(t);
  cta.meet(v);
}
inline uint32_t __shfl_sync(unsigned mask, uint32_t x, int src, int width = 32) {
  cta.word[threadIdx.x] = x;
  cta.meet(lanes(mask));
  const uint32_t r = cta.word[(threadIdx.x & ~(unsigned)(width - 1)) + src];
  cta.meet(lanes(mask));
  return r;
}
// named by kernels that are not run here
template <class V> V __shfl_up_sync(unsigned, V x, int) { return x; }
template <class V> V __shfl_xor_sync(unsigned, V x, int) { return x; }
inline int __syncthreads_or(int x) { return x; }
template <class V> V atomicAdd(V* p, V x) { const V o = *p; *p += x; return o; }
inline int atomicCAS(int* p, int, int) { return *p; }

#include "msm.cuh"

// one row of 2^m elements: R and S, X | Y | Z of N words each, in place
template <class C>
int tree(int m, uint32_t* R, uint32_t* S) {
  using F = typename C::Fp;
  static_assert(ecc::kJacThreads == T, "");
  const size_t n = (size_t)1 << m, bytes = n * sizeof(ecc::Jac<F>);
  std::vector<uint4> r(bytes / 16), s(bytes / 16);
  std::memcpy(r.data(), R, bytes);
  std::memcpy(s.data(), S, bytes);
  ecc::MsmInst in{};
  in.c = (uint32_t)m + 1;
  in.Wr = 1;
  ecc::RedArgs<C> a{};
  a.inst = &in;
  a.num = 1;
  a.elems = n;
  a.R = reinterpret_cast<ecc::Jac<F>*>(r.data());
  a.S = reinterpret_cast<ecc::Jac<F>*>(s.data());
  cta.stuck = false;
  for (int t = 0; t < T; ++t) cta.state[t] = READY;
  cta.run = 0;
  std::vector<std::thread> th;
  for (int t = 0; t < T; ++t)
    th.emplace_back([&, t] {
      threadIdx.x = t;
      blockIdx.x = 0;
      try {
        {
          std::unique_lock<std::mutex> l(cta.mu);
          cta.wait_turn(l, t);
        }
        ecc::k_msm_tree<C>(a, 0);
      } catch (Stuck&) {
      }
      std::unique_lock<std::mutex> l(cta.mu);
      cta.state[t] = DONE;
      if (!cta.stuck) cta.next();
    });
  for (auto& t : th) t.join();
  std::memcpy(R, r.data(), bytes);
  std::memcpy(S, s.data(), bytes);
  return cta.stuck ? 1 : 0;
}
extern "C" int run_tree(int curve, int m, uint32_t* R, uint32_t* S) {
  return curve == 2 ? tree<ecc::BN254>(m, R, S) : tree<ecc::BLS12_381>(m, R, S);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tree")
    for f in os.listdir(CSRC):
        if f.endswith(".cuh"):
            shutil.copy(os.path.join(CSRC, f), d / f)
    (d / "ptx.cuh").write_text(PTX)
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-pthread", "-shared", "-fPIC", f"-I{d}", str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


def _pack(C, pts, zs):
    """Jacobian Montgomery words of points (None: O), each with its own Z."""
    r = 1 << (32 * C.limbs)
    rows = []
    for P, z in zip(pts, zs):
        xyz = (1, 1, 0) if P is None else (P[0] * z * z % C.p, P[1] * z ** 3 % C.p, z)
        rows.append(np.concatenate([synth.ints_to_limbs([v * r % C.p], C.limbs)[0] for v in xyz]))
    return np.ascontiguousarray(np.stack(rows).astype(np.uint32))


def _unpack(C, words):
    ri = pow(1 << (32 * C.limbs), -1, C.p)
    out = []
    for row in words.reshape(-1, 3, C.limbs):
        x, y, z = (synth.limbs_to_int(v) * ri % C.p for v in row)
        zi = pow(z, -1, C.p) if z else 0
        out.append((x * zi * zi % C.p, y * zi ** 3 % C.p) if z else None)
    return out


@pytest.mark.parametrize("cid", [2, 3])
@pytest.mark.parametrize("m", [1, 4])
def test_lanes_that_run_ahead(lib, cid, m):
    """Elements O (empty buckets), equal, opposite and plain; after the levels R[0] and
    S[0] are the row's sums and R[2^j] the sum of the elements whose index has bit j."""
    C, n = curves.BY_ID[cid], 1 << m
    P = [ec.mul(C, 5 + 3 * i, C.G) for i in range(n)]
    for i, v in ((0, None), (3, ec.neg(C, ec.mul(C, 11, C.G))), (5, ec.mul(C, 17, C.G)), (6, None), (7, None)):
        if i < n:
            P[i] = v
    Q = list(reversed(P))
    R, S = _pack(C, P, range(2, n + 2)), _pack(C, Q, range(7, n + 7))
    word = ctypes.POINTER(ctypes.c_uint32)
    assert lib.run_tree(cid, m, R.ctypes.data_as(word), S.ctypes.data_as(word)) == 0, "lanes wait for lanes that are gone"

    def total(pts):
        acc = None
        for p in pts:
            acc = ec.add(C, acc, p)
        return acc

    got, got_s = _unpack(C, R), _unpack(C, S)
    assert got[0] == total(P) and got_s[0] == total(Q)
    for j in range(m):
        assert got[1 << j] == total(p for i, p in enumerate(P) if i >> j & 1)
