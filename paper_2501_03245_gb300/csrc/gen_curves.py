#!/usr/bin/env python3
"""Writes curves_gen.cuh: compile-time constants of the four curves for the CUDA
library (moduli, Montgomery constants R mod q, R^2 mod q, -q^-1 mod 2^32, q-2,
curve coefficients in Montgomery form, generators).

Run from this directory: ``python gen_curves.py`` (the output is committed).
The parameters are the published standard ones: SEC 2 (secp256k1,
secp256r1 = NIST P-256), the BN254 polynomial in u = 0x44E992B44A6909F1 with
b = 3 and generator (1, 2), and BLS12-381 (x = -0xd201000000010000, b = 4, the
standard G1 generator), and the SM2 recommended curve of GB/T 32918.5.
"""
import os

CURVES = [
    # name, field prime p, a, b, Gx, Gy, group order n
    ("Secp256k1",
     0xFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFEFFFFFC2F, 0, 7,
     0x79BE667EF9DCBBAC55A06295CE870B07029BFCDB2DCE28D959F2815B16F81798,
     0x483ADA7726A3C4655DA4FBFC0E1108A8FD17B448A68554199C47D08FFB10D4B8,
     0xFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFEBAAEDCE6AF48A03BBFD25E8CD0364141),
    ("P256",
     0xFFFFFFFF00000001000000000000000000000000FFFFFFFFFFFFFFFFFFFFFFFF, -3,
     0x5AC635D8AA3A93E7B3EBBD55769886BC651D06B0CC53B0F63BCE3C3E27D2604B,
     0x6B17D1F2E12C4247F8BCE6E563A440F277037D812DEB33A0F4A13945D898C296,
     0x4FE342E2FE1A7F9B8EE7EB4A7C0F9E162BCE33576B315ECECBB6406837BF51F5,
     0xFFFFFFFF00000000FFFFFFFFFFFFFFFFBCE6FAADA7179E84F3B9CAC2FC632551),
    ("BN254",
     0x30644E72E131A029B85045B68181585D97816A916871CA8D3C208C16D87CFD47, 0, 3, 1, 2,
     0x30644E72E131A029B85045B68181585D2833E84879B9709143E1F593F0000001),
    ("BLS12_381",
     0x1A0111EA397FE69A4B1BA7B6434BACD764774B84F38512BF6730D2A0F6B0F6241EABFFFEB153FFFFB9FEFFFFFFFFAAAB,
     0, 4,
     0x17F1D3A73197D7942695638C4FA9AC0FC3688C4F9774B905A14E3A3F171BAC586C55E83FF97A1AEFFB3AF00ADB22C6BB,
     0x08B3F481E3AAA0F1A09E30ED741D8AE4FCF5E095D5D00AF600DB18CB2C04B3EDD03CC744A2888AE40CAA232946C5E7E1,
     0x73EDA753299D7D483339D80809A1D80553BDA402FFFE5BFEFFFFFFFF00000001),
    ("SM2",
     0xFFFFFFFEFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFF00000000FFFFFFFFFFFFFFFF, -3,
     0x28E9FA9E9D9F5E344D5A9E4BCF6509A7F39789F515AB8F92DDBCBD414D940E93,
     0x32C4AE2C1F1981195F9904466A39C9948FE30BBFF2660BE1715A4589334C74C7,
     0xBC3736A2F4F6779C59BDCEE36B692153D0A9877CC62A474002DF32E52139F0A0,
     0xFFFFFFFEFFFFFFFFFFFFFFFFFFFFFFFF7203DF6B21C6052B53BBF40939D54123),
]


# Moduli whose multiplication uses the shape of the prime (fp.cuh): FORM 1 is the
# NIST P-256 prime 2^256 - 2^224 + 2^192 + 2^96 - 1, FORM 2 the secp256k1 prime
# 2^256 - 2^32 - 977 (elements held as plain integers: R = 1), FORM 3 the SM2
# prime 2^256 - 2^224 - 2^96 + 2^64 - 1.  Each also gets a class <name>Mont with
# the generic Montgomery multiplication, which the probes compare with.
FORMS = {
    0xFFFFFFFF00000001000000000000000000000000FFFFFFFFFFFFFFFFFFFFFFFF: 1,
    (1 << 256) - (1 << 32) - 977: 2,
    (1 << 256) - (1 << 224) - (1 << 96) + (1 << 64) - 1: 3,
}


def limbs(v, n):
    return [(v >> (32 * i)) & 0xFFFFFFFF for i in range(n)]


def arr(name, v, n):
    """A constexpr limb accessor: name(i) is limb i (0 outside the range)."""
    cases = " ".join(f"case {i}: return 0x{x:08x}u;" for i, x in enumerate(limbs(v, n)))
    return (f"  ECC_DEV static constexpr uint32_t {name}(int i) {{\n"
            f"    switch (i) {{ {cases} default: return 0u; }}\n  }}\n")


def traits(name, q, form):
    n = (q.bit_length() + 31) // 32
    n += n % 2  # even limb count for the even/odd carry chains
    R = 1 if form == 2 else 1 << (32 * n)
    qinv = (-pow(q, -1, 1 << 32)) % (1 << 32)
    s = f"struct {name} {{\n"
    s += f"  static constexpr int N = {n};\n"
    s += f"  static constexpr int BITS = {q.bit_length()};\n"
    s += f"  static constexpr uint32_t QINV = 0x{qinv:08x}u;\n"
    s += f"  static constexpr int FORM = {form};\n"
    s += f"  static constexpr bool SQR_ROWS = {'true' if q.bit_length() < 32 * n else 'false'};\n"
    s += f"  static constexpr uint64_t QINV62 = 0x{pow(q, -1, 1 << 62):016x}ull;  // q^-1 mod 2^62\n"
    s += "  ECC_DEV static constexpr uint32_t qinv() { return QINV; }\n"
    s += "  ECC_DEV static constexpr uint64_t qinv62() { return QINV62; }\n"
    s += arr("p", q, n) + arr("r2", R * R % q, n) + arr("one", R % q, n) + arr("pm2", q - 2, n)
    s += arr("r3", R * R * R % q, n)
    s += "};\n\n"
    return s, n, R


def field(name, q):
    form = FORMS.get(q, 0)
    s, n, R = traits(name, q, form)
    if form == 2:
        s += traits(name + "Mont", q, 0)[0]
    elif form:
        s += f"struct {name}Mont : {name} {{\n  static constexpr int FORM = 0;\n}};\n\n"
    return s, n, R


# The endomorphism (x, y) -> (beta x, y) of the curves with a = 0 multiplies the points
# of a group of prime order by lambda, beta and lambda cube roots of unity mod p and mod
# n (Gallant, Lambert and Vanstone, "Faster point multiplication on elliptic curves with
# efficient endomorphisms", CRYPTO 2001).  Only for groups that are the whole curve
# (cofactor 1), where every point on the curve is such a point.
GLV = ("Secp256k1", "BN254")
GLV_SHIFT = 320


def cube_root(q):
    g = 2
    while pow(g, (q - 1) // 3, q) == 1:
        g += 1
    return pow(g, (q - 1) // 3, q)


def times(k, x, y, p):
    """k (x, y) on y^2 = x^3 + b, affine; k > 0 below the order."""
    rx = None
    for bit in bin(k)[2:]:
        if rx is not None:
            m = 3 * rx * rx * pow(2 * ry, -1, p) % p
            nx = (m * m - 2 * rx) % p
            rx, ry = nx, (m * (rx - nx) - ry) % p
        if bit == "1":
            if rx is None:
                rx, ry = x, y
            else:
                m = (ry - y) * pow(rx - x, -1, p) % p
                nx = (m * m - rx - x) % p
                rx, ry = nx, (m * (x - nx) - y) % p
    return rx, ry


def glv(p, n, gx, gy, R, N):
    """Constants that write k as k1 + k2 lambda with short k1, k2: with a basis (a1, b1),
    (a2, b2) of the lattice of a + b lambda = 0 mod n, c1 = round(b2 k / n), c2 =
    round(-b1 k / n), k1 = k - c1 a1 - c2 a2, k2 = -c1 b1 - c2 b2.  c_i comes from k times
    g_i = 2^320 |b| / n; the signs are in the other factors (mod 2^160)."""
    lam, beta = cube_root(n), cube_root(p)
    lx, ly = times(lam, gx, gy, p)
    assert ly == gy
    if lx != beta * gx % p:
        beta = beta * beta % p
    assert lx == beta * gx % p
    # half-extended Euclid on (n, lambda): the remainders around sqrt(n)
    rows, (r0, t0), (r1, t1) = [], (n, 0), (lam, 1)
    while r1:
        rows.append((r1, -t1))
        q = r0 // r1
        (r0, t0), (r1, t1) = (r1, t1), (r0 - q * r1, t0 - q * t1)
    i = next(j for j, (r, _) in enumerate(rows) if r * r < n)
    (a1, b1), (a2, b2) = sorted(rows[i - 1:i + 2], key=lambda v: v[0] ** 2 + v[1] ** 2)[:2]
    if a1 * b2 - a2 * b1 < 0:
        (a1, b1), (a2, b2) = (a2, b2), (a1, b1)
    assert a1 * b2 - a2 * b1 == n and (a1 + b1 * lam) % n == 0 and (a2 + b2 * lam) % n == 0
    bits = max(abs(a1) + abs(a2), abs(b1) + abs(b2)) // 2 + 1
    s1, s2 = (1 if b2 > 0 else -1), (1 if -b1 > 0 else -1)
    g = [((abs(v) << GLV_SHIFT) + n // 2) // n for v in (b2, b1)]
    assert max(g) < 1 << 224
    m = 1 << 160
    s = "  static constexpr bool GLV = true;\n"
    s += f"  static constexpr int GLV_BITS = {bits.bit_length()};  // |k1|, |k2| < 2^GLV_BITS\n"
    s += arr("glv_beta", beta * R % p, N) + arr("glv_g1", g[0], 7) + arr("glv_g2", g[1], 7)
    s += arr("glv_a1", -s1 * a1 % m, 5) + arr("glv_a2", -s2 * a2 % m, 5)
    s += arr("glv_b1", -s1 * b1 % m, 5) + arr("glv_b2", -s2 * b2 % m, 5)
    return s


def main():
    out = ["// Generated by gen_curves.py; do not edit.\n#pragma once\n#include <cstdint>\n",
           "#ifndef ECC_DEV\n#define ECC_DEV __device__ __forceinline__\n#endif\n\n",
           "namespace ecc {\n\n"]
    for name, p, a, b, gx, gy, n in CURVES:
        fs, N, R = field(f"{name}Fp", p)
        ns, NN, RN = field(f"{name}Fn", n)
        out.append(fs)
        out.append(ns)
        a %= p
        s = f"struct {name} {{\n"
        s += f"  using Fp = {name}Fp;\n  using Fn = {name}Fn;\n"
        s += f"  static constexpr bool A_ZERO = {'true' if a == 0 else 'false'};\n"
        s += arr("a", a * R % p, N) + arr("b", b * R % p, N)
        s += arr("gx", gx, N) + arr("gy", gy, N)
        s += arr("n", n, 8)
        s += f"  static constexpr int SCALAR_BITS = {n.bit_length()};\n"
        s += glv(p, n, gx, gy, R, N) if name in GLV else "  static constexpr bool GLV = false;\n"
        s += "};\n\n"
        out.append(s)
    out.append("}  // namespace ecc\n")
    here = os.path.dirname(os.path.abspath(__file__))
    with open(os.path.join(here, "curves_gen.cuh"), "w") as f:
        f.write("".join(out))


if __name__ == "__main__":
    main()
