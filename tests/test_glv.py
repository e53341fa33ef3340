"""The endomorphism's scalar split (glv.cuh), compiled for the host: k1 + k2 lambda = k
mod n, both below the declared length, for random scalars and the edges of the range;
beta and lambda belong together on the curve."""
import ctypes
import os
import random
import subprocess

import pytest

from oracle import curves, ec

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_03245_gb300", "csrc")
SRC = """
#define ECC_DEV inline
#include <cstdint>
#include "glv.cuh"
template <class C> static int run(const uint32_t* k, uint32_t* m, uint32_t* beta) {
  bool n1, n2;
  ecc::glv_split<C>(k, m, n1, m + 5, n2);
  for (int i = 0; i < 8; ++i) beta[i] = C::glv_beta(i);
  return (n1 ? 1 : 0) | (n2 ? 2 : 0) | (C::GLV_BITS << 2);
}
extern "C" int split(int curve, const uint32_t* k, uint32_t* m, uint32_t* beta) {
  return curve == 0 ? run<ecc::Secp256k1>(k, m, beta) : run<ecc::BN254>(k, m, beta);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("glv")
    src, so = d / "s.cpp", d / "s.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-shared", "-fPIC", f"-I{CSRC}", str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("cid", [0, 2])
def test_split(lib, cid):
    C = curves.BY_ID[cid]
    k8, m10, b8 = (ctypes.c_uint32 * 8)(), (ctypes.c_uint32 * 10)(), (ctypes.c_uint32 * 8)()

    def split(k):
        for i in range(8):
            k8[i] = (k >> (32 * i)) & 0xFFFFFFFF
        f = lib.split(cid, k8, m10, b8)
        v = [sum(m10[5 * h + i] << (32 * i) for i in range(5)) for h in range(2)]
        assert max(v) < 1 << (f >> 2)
        return (-v[0] if f & 1 else v[0]), (-v[1] if f & 2 else v[1])

    split(0)
    beta = sum(b8[i] << (32 * i) for i in range(8))
    if cid == 2:  # Montgomery form; the secp256k1 field is held as plain integers
        beta = beta * pow(1 << 256, -1, C.p) % C.p
    assert beta != 1 and pow(beta, 3, C.p) == 1
    lams = [x for x in (pow(g, (C.n - 1) // 3, C.n) for g in range(2, 12)) if x != 1]
    lam = next(x for x in lams if ec.mul(C, x, C.G) == (beta * C.G[0] % C.p, C.G[1]))
    rnd = random.Random(7 + cid)
    ks = [0, 1, 2, C.n - 1, C.n - 2, C.n // 2, C.n // 2 + 1, lam, lam - 1, lam + 1, C.n - lam]
    ks += [rnd.randrange(C.n) for _ in range(20000)]
    ks += [(1 << e) % C.n for e in range(256)] + [C.n - 1 - ((1 << e) % C.n) for e in range(255)]
    ks += [(a + b * lam) % C.n for a in (0, 1, 1 << 63, (1 << 126) - 1) for b in (0, 1, 1 << 63, (1 << 126) - 1)]
    for k in ks:
        k1, k2 = split(k)
        assert (k1 + k2 * lam - k) % C.n == 0
