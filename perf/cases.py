"""Timed cases of the library: what its users have it do, through the entry points.

A case is a plain dict.  ``prepare`` makes a user's inputs on the GPU (signed
triples, points, scalars, resident bases), ``run`` is one call of the entry point,
``work`` counts the bytes and operations of the textbook method and ``exact`` gives
the results from Python integers where that is quick.

One operation ("flop") of ``work`` is half a 32-bit wide multiply-add; a modular
multiplication of m limbs is 2 m^2 + m of those.
"""
import math

import numpy as np
import torch

from paper_2501_03245_gb300 import ecc

# name -> (id, p, a, b, Gx, Gy, group order, limbs of a base-field element)
_P256 = 2**256 - 2**224 + 2**192 + 2**96 - 1
_SM2 = 2**256 - 2**224 - 2**96 + 2**64 - 1
_U, _X = 0x44E992B44A6909F1, -0xD201000000010000
_BLS_R = _X**4 - _X**2 + 1
CURVES = {
    "secp256k1": (ecc.ECC_SECP256K1, 2**256 - 2**32 - 977, 0, 7,
                  0x79BE667EF9DCBBAC55A06295CE870B07029BFCDB2DCE28D959F2815B16F81798,
                  0x483ADA7726A3C4655DA4FBFC0E1108A8FD17B448A68554199C47D08FFB10D4B8,
                  0xFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFFEBAAEDCE6AF48A03BBFD25E8CD0364141, 8),
    "P-256": (ecc.ECC_P256, _P256, _P256 - 3, 0x5AC635D8AA3A93E7B3EBBD55769886BC651D06B0CC53B0F63BCE3C3E27D2604B,
              0x6B17D1F2E12C4247F8BCE6E563A440F277037D812DEB33A0F4A13945D898C296,
              0x4FE342E2FE1A7F9B8EE7EB4A7C0F9E162BCE33576B315ECECBB6406837BF51F5,
              0xFFFFFFFF00000000FFFFFFFFFFFFFFFFBCE6FAADA7179E84F3B9CAC2FC632551, 8),
    "BN254": (ecc.ECC_BN254, 36 * _U**4 + 36 * _U**3 + 24 * _U**2 + 6 * _U + 1, 0, 3, 1, 2,
              36 * _U**4 + 36 * _U**3 + 18 * _U**2 + 6 * _U + 1, 8),
    "BLS12-381": (ecc.ECC_BLS12_381, (_X - 1) ** 2 * _BLS_R // 3 + _X, 0, 4,
                  0x17F1D3A73197D7942695638C4FA9AC0FC3688C4F9774B905A14E3A3F171BAC586C55E83FF97A1AEFFB3AF00ADB22C6BB,
                  0x08B3F481E3AAA0F1A09E30ED741D8AE4FCF5E095D5D00AF600DB18CB2C04B3EDD03CC744A2888AE40CAA232946C5E7E1,
                  _BLS_R, 12),
    "SM2": (ecc.ECC_SM2, _SM2, _SM2 - 3, 0x28E9FA9E9D9F5E344D5A9E4BCF6509A7F39789F515AB8F92DDBCBD414D940E93,
            0x32C4AE2C1F1981195F9904466A39C9948FE30BBFF2660BE1715A4589334C74C7,
            0xBC3736A2F4F6779C59BDCEE36B692153D0A9877CC62A474002DF32E52139F0A0,
            0xFFFFFFFEFFFFFFFFFFFFFFFFFFFFFFFF7203DF6B21C6052B53BBF40939D54123, 8),
}
SIGNING = ("secp256k1", "P-256", "SM2")
PAIRING = ("BN254", "BLS12-381")


def listed():
    return [
        # one signature as it arrives: launches and latency are all there is
        {"name": "verify_one", "kind": "verify", "curve": "secp256k1", "n": 1},
        # a block of transactions
        {"name": "verify_block", "kind": "verify", "curve": "secp256k1", "n": 4096},
        # a queue that has been drained: an odd number of signatures
        {"name": "verify_queue", "kind": "verify", "curve": "SM2", "n": 50021},
        # a full batch, the throughput a verification service is sized by
        {"name": "verify_batch", "kind": "verify", "curve": "P-256", "n": 1 << 20},
        # a full batch of signatures with their public keys
        {"name": "sign_batch", "kind": "sign", "curve": "SM2", "n": 1 << 20},
        # key generation k G for an odd number of keys
        {"name": "keygen", "kind": "fpmul", "curve": "P-256", "n": 100003},
        # a small commitment, points and scalars handed over with the call
        {"name": "msm_small", "kind": "msm", "curve": "BN254", "n": 4096},
        # a commitment of a mid-sized circuit, an odd number of points
        {"name": "msm_odd", "kind": "msm", "curve": "BLS12-381", "n": 130003},
        # a ragged batch of commitments in one call
        {"name": "msm_ragged", "kind": "msm_ragged", "curve": "BN254", "num": 256, "lo": 10, "hi": 18, "sizes": 7},
        # a prover's resident bases with window multiples, many vectors a call
        {"name": "msm_bases", "kind": "msm_bases", "curve": "BLS12-381", "n": 1 << 20, "vectors": 16, "c": 20},
        # additions of two arrays of points (trees of commitments, key aggregation)
        {"name": "point_add", "kind": "point_add", "curve": "BN254", "n": 262147},
        # inverses of an array of scalars (Lagrange and barycentric coefficients)
        {"name": "inv_batch", "kind": "fp", "curve": "BLS12-381", "op": "inv_batch", "field": 1, "n": 1000003},
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [2^lo, 2^hi]."""
    return int(2 ** rng.uniform(lo, hi))


def draw(rng):
    kind = rng.choice(["verify", "verify", "verify", "sign", "fpmul", "msm", "msm", "msm_ragged", "msm_bases",
                       "msm_bases", "point_add", "point_dbl", "fp"])
    if kind in ("verify", "sign"):
        return {"kind": kind, "curve": rng.choice(SIGNING), "n": _log(rng, 0, 20)}
    if kind in ("fpmul", "point_add", "point_dbl"):
        return {"kind": kind, "curve": rng.choice(sorted(CURVES)), "n": _log(rng, 4, 20)}
    if kind == "fp":
        op = rng.choice(["mul", "add", "inv", "inv_batch"])
        return {"kind": "fp", "curve": rng.choice(sorted(CURVES)), "op": op, "field": rng.randrange(2),
                "n": _log(rng, 8, 20)}
    if kind == "msm":
        return {"kind": kind, "curve": rng.choice(PAIRING), "n": _log(rng, 8, 20)}
    if kind == "msm_ragged":
        lo = rng.randint(8, 12)
        return {"kind": kind, "curve": rng.choice(PAIRING), "num": _log(rng, 1, 7), "lo": lo,
                "hi": lo + rng.randint(2, 6), "sizes": rng.randrange(1 << 20)}
    n = _log(rng, 12, 20)
    vectors = min(_log(rng, 0, 4), (1 << 22) // n + 1)
    c = rng.choice([0, max(10, min(20, int(math.log2(n * vectors)) - 1))])
    return {"kind": kind, "curve": rng.choice(PAIRING), "n": n, "vectors": vectors, "c": c}


# ------------------------------------------------------------------ inputs


def _below(rng, n, bound, limbs):
    """n integers spread over [0, bound) as little-endian 32-bit limbs."""
    a = rng.integers(0, 1 << 32, size=(n, limbs), dtype=np.uint32)
    top = (bound - 1) >> (32 * (limbs - 1))
    a[:, limbs - 1] = rng.integers(0, top, size=n, dtype=np.uint32)
    return a


def _bytes(a):
    """Limbs as big-endian bytes."""
    return np.ascontiguousarray(a[:, ::-1]).astype(">u4").view(np.uint8).reshape(a.shape[0], 4 * a.shape[1])


def _gpu(a):
    return torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda()


def _rng(seed):
    return np.random.Generator(np.random.SFC64(seed))


def _ecdsa_inputs(case, seed):
    """Keys, hashes and nonces, and which signatures get one bit of r or s flipped: 1/16 of
    them, and the first one for every other seed, so that a single one is met both ways."""
    n, order, rng = case["n"], CURVES[case["curve"]][6], _rng(seed)
    d, e, k = (_bytes(_below(rng, n, order, 8)) for _ in range(3))
    flip = rng.integers(0, 16, size=n) == 0
    flip[0] = seed % 2 == 1
    bad = np.flatnonzero(flip)
    return d, e, k, bad, rng.integers(0, 2, size=bad.size), rng.integers(0, 256, size=bad.size)


def _sizes(case):
    if case["kind"] != "msm_ragged":
        return None
    u = np.random.default_rng(case["sizes"]).random(case["num"])
    return np.floor(np.exp2(case["lo"] + (case["hi"] - case["lo"]) * u)).astype(np.int64)


def _msm_inputs(case, seed):
    """Multipliers of the points a_i G, and the scalars."""
    order, rng = CURVES[case["curve"]][6], _rng(seed)
    n = int(_sizes(case).sum()) if case["kind"] == "msm_ragged" else case["n"]
    return _below(rng, n, order, 8), _below(rng, n * case.get("vectors", 1), order, 8)


def _multiples(cid, limbs, a):
    out = torch.empty((a.shape[0], 2 * limbs), dtype=torch.int32, device="cuda")
    ecc.ecc_fixed_base_mul(cid, a.shape[0], _gpu(a), out)
    return out


class _Bases:
    """Resident bases, given back with the state."""

    def __init__(self, cid, n, points, c):
        self.handle = ecc.ecc_bases_create(cid, n, points)
        if c:
            ecc.ecc_bases_precompute(self.handle, c)

    def __del__(self):
        torch.cuda.synchronize()
        ecc.ecc_bases_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    cid, p, _, _, _, _, order, m = CURVES[case["curve"]]
    st = {"case": case, "cid": cid}
    if kind in ("verify", "sign"):
        n = case["n"]
        d, e, k, bad, which, bit = _ecdsa_inputs(case, seed)
        d, e, k = _gpu(d), _gpu(e), _gpu(k)
        r, s = (torch.empty((n, 32), dtype=torch.uint8, device="cuda") for _ in range(2))
        pub = torch.empty((n, 64), dtype=torch.uint8, device="cuda")
        if kind == "sign":
            st.update(d=d, e=e, k=k, r=r, s=s, pub=pub)
            return st
        ecc.ecc_sign_batch(cid, n, d, e, k, r, s, pub)
        mask = (1 << (bit % 8)).astype(np.uint8)
        for buf, w in ((r, 0), (s, 1)):
            i = torch.from_numpy(bad[which == w]).cuda()
            j = torch.from_numpy(31 - bit[which == w] // 8).cuda()
            buf[i, j] ^= torch.from_numpy(mask[which == w]).cuda()
        st.update(e=e, r=r, s=s, pub=pub, ok=torch.empty(n, dtype=torch.uint8, device="cuda"))
    elif kind == "fpmul":
        st["k"] = _gpu(_below(_rng(seed), case["n"], order, 8))
        st["out"] = torch.empty((case["n"], 2 * m), dtype=torch.int32, device="cuda")
    elif kind in ("point_add", "point_dbl"):
        rng = _rng(seed)
        st["p"], st["q"] = (_multiples(cid, m, _below(rng, case["n"], order, 8)) for _ in range(2))
        st["out"] = torch.empty_like(st["p"])
    elif kind == "fp":
        q, limbs = (order, 8) if case["field"] else (p, m)
        rng = _rng(seed)
        st["a"], st["b"] = (_gpu(_below(rng, case["n"], q, limbs)) for _ in range(2))
        st["out"] = torch.empty_like(st["a"])
    else:
        a, k = _msm_inputs(case, seed)
        points, st["k"] = _multiples(cid, m, a), _gpu(k)
        rows = case["num"] if kind == "msm_ragged" else case.get("vectors", 1)
        st["out"] = torch.empty((rows, 2 * m), dtype=torch.int32, device="cuda")
        if kind == "msm_bases":
            st["bases"] = _Bases(cid, case["n"], points, case["c"])
        else:
            st["points"] = points
        if kind == "msm_ragged":
            st["offsets"] = np.concatenate([[0], np.cumsum(_sizes(case))]).astype(np.uint64)
    return st


def run(st):
    case, cid = st["case"], st["cid"]
    kind = case["kind"]
    if kind == "verify":
        ecc.ecc_verify_batch(cid, case["n"], st["e"], st["r"], st["s"], st["pub"], st["ok"])
        return st["ok"]
    if kind == "sign":
        ecc.ecc_sign_batch(cid, case["n"], st["d"], st["e"], st["k"], st["r"], st["s"], st["pub"])
        return {"r": st["r"], "s": st["s"], "pub": st["pub"]}
    if kind == "fpmul":
        ecc.ecc_fixed_base_mul(cid, case["n"], st["k"], st["out"])
    elif kind == "point_add":
        ecc.ecc_point_add_batch(cid, case["n"], st["p"], st["q"], st["out"])
    elif kind == "point_dbl":
        ecc.ecc_point_dbl_batch(cid, case["n"], st["p"], st["out"])
    elif kind == "msm":
        ecc.ecc_msm(cid, case["n"], st["points"], st["k"], st["out"])
    elif kind == "msm_ragged":
        ecc.ecc_msm_ragged(cid, case["num"], st["offsets"], st["points"], st["k"], st["out"])
    elif kind == "msm_bases":
        ecc.ecc_msm_bases(st["bases"].handle, case["vectors"], st["k"], st["out"])
    elif case["op"] in ("mul", "add"):
        fn = ecc.ecc_fp_mul if case["op"] == "mul" else ecc.ecc_fp_add
        fn(cid, case["field"], case["n"], st["a"], st["b"], st["out"])
    else:
        fn = ecc.ecc_fp_inv if case["op"] == "inv" else ecc.ecc_fp_inv_batch
        fn(cid, case["field"], case["n"], st["a"], st["out"])
    return st["out"]


# ------------------------------------------------------------------ work


def work(case):
    """Inputs read once and outputs written once; modular multiplications of the
    textbook method (6 per batched affine addition, 7 per doubling)."""
    kind, n, m = case["kind"], case.get("n", 0), CURVES[case["curve"]][7]
    bits = CURVES[case["curve"]][6].bit_length()

    def bucket(size):
        # signed windows of the best width: 6 a digit, 12 a bucket, the combination
        return min(6 * size * -(-(bits + 1) // c) + -(-(bits + 1) // c) * (12 * 2 ** (c - 1) + 7 * c)
                   for c in range(2, 21))

    if kind == "verify":
        nbytes, muls = n * (32 * 3 + 64 + 1), n * 2405
    elif kind == "sign":
        nbytes, muls = n * (32 * 3 + 32 * 2 + 64), n * 391
    elif kind == "fpmul":
        nbytes, muls = n * (32 + 8 * m), n * 192
    elif kind in ("point_add", "point_dbl"):
        nbytes, muls = n * 8 * m * (3 if kind == "point_add" else 2), n * (6 if kind == "point_add" else 7)
    elif kind == "fp":
        m = 8 if case["field"] else m
        nbytes = n * 4 * m * (3 if case["op"] in ("mul", "add") else 2)
        muls = n * {"mul": 1, "add": 0, "inv": 3, "inv_batch": 3}[case["op"]]
    elif kind == "msm_ragged":
        sizes = [int(s) for s in _sizes(case)]
        nbytes, muls = sum(sizes) * (32 + 8 * m) + len(sizes) * 8 * m, sum(bucket(s) for s in sizes)
    elif kind == "msm_bases" and case["c"]:
        v, c = case["vectors"], case["c"]
        windows = -(-(bits + 1) // c)
        nbytes = v * n * 32 + windows * n * 8 * m
        muls = v * (6 * n * windows + 12 * 2 ** (c - 1))
    else:
        v = case.get("vectors", 1)
        nbytes, muls = v * n * 32 + n * 8 * m + v * 8 * m, v * bucket(n)
    return {"bytes": nbytes, "flops": 2 * muls * (2 * m * m + m) + (n * m if kind == "fp" else 0)}


# ------------------------------------------------------------------ exact values


def _ints(a):
    raw, w = np.ascontiguousarray(a).tobytes(), 4 * a.shape[1]
    return [int.from_bytes(raw[i:i + w], "little") for i in range(0, len(raw), w)]


def _limbs(vals, m):
    raw = b"".join(v.to_bytes(4 * m, "little") for v in vals)
    return np.frombuffer(raw, dtype=np.int32).reshape(len(vals), m).copy()


def _inverses(vals, q):
    """Inverses mod q of a list (0 for 0) with one modular inversion."""
    pre, run = [], 1
    for v in vals:
        pre.append(run)
        run = run * (v or 1) % q
    inv, out = pow(run, -1, q), [0] * len(vals)
    for i in range(len(vals) - 1, -1, -1):
        out[i] = inv * pre[i] % q if vals[i] else 0
        inv = inv * (vals[i] or 1) % q
    return out


def _times_g(curve, k):
    """k G as affine integers, (0, 0) for the point at infinity (Jacobian double and add)."""
    _, p, a, _, gx, gy, order, _ = CURVES[curve]
    x, y, z = 0, 1, 0
    for bit in bin(k % order)[2:]:
        if z:
            s, w = 4 * x * y * y % p, (3 * x * x + a * pow(z, 4, p)) % p
            x2 = (w * w - 2 * s) % p
            x, y, z = x2, (w * (s - x2) - 8 * pow(y, 4, p)) % p, 2 * y * z % p
        if bit == "1":
            if not z:
                x, y, z = gx, gy, 1
                continue
            zz = z * z % p
            h, r = (gx * zz - x) % p, (gy * zz * z - y) % p
            if h == 0:
                if r:
                    x, y, z = 0, 1, 0
                    continue
                s, w = 4 * x * y * y % p, (3 * x * x + a * pow(z, 4, p)) % p
                x2 = (w * w - 2 * s) % p
                x, y, z = x2, (w * (s - x2) - 8 * pow(y, 4, p)) % p, 2 * y * z % p
                continue
            hh = h * h % p
            hhh, v = h * hh % p, x * hh % p
            x3 = (r * r - hhh - 2 * v) % p
            x, y, z = x3, (r * (v - x3) - y * hhh) % p, z * h % p
    if not z:
        return 0, 0
    zi = pow(z, -1, p)
    return x * zi * zi % p, y * zi * zi * zi % p


def _points(curve, ks):
    m = CURVES[curve][7]
    pts = [_times_g(curve, k) for k in ks]
    return np.concatenate([_limbs([q[0] for q in pts], m), _limbs([q[1] for q in pts], m)], axis=1)


def _dot(a, k):
    """sum_i a_i k_i of two limb arrays (sums of 2^20 products of 16-bit digits are exact in doubles)."""
    total = 0
    for lo in range(0, a.shape[0], 1 << 20):
        x = np.ascontiguousarray(a[lo:lo + (1 << 20)]).view(np.uint16).astype(np.float64)
        y = np.ascontiguousarray(k[lo:lo + (1 << 20)]).view(np.uint16).astype(np.float64)
        z = x.T @ y
        total += sum(int(z[i, j]) << (16 * (i + j)) for i in range(z.shape[0]) for j in range(z.shape[1]))
    return total


def exact(case, seed):
    kind, curve = case["kind"], case["curve"]
    _, p, _, _, _, _, order, m = CURVES[curve]
    if kind == "verify":  # a signature is valid unless a bit of it was flipped
        ok = np.ones(case["n"], dtype=np.uint8)
        ok[_ecdsa_inputs(case, seed)[3]] = 0
        return ok
    if kind == "fp":
        q, limbs = (order, 8) if case["field"] else (p, m)
        rng = _rng(seed)
        a, b = (_ints(_below(rng, case["n"], q, limbs)) for _ in range(2))
        if case["op"] == "mul":
            return _limbs([x * y % q for x, y in zip(a, b)], limbs)
        if case["op"] == "add":
            return _limbs([(x + y) % q for x, y in zip(a, b)], limbs)
        return _limbs(_inverses(a, q), limbs)
    if kind in ("fpmul", "point_add", "point_dbl"):
        if case["n"] > 1000:
            return None
        rng = _rng(seed)
        a = _ints(_below(rng, case["n"], order, 8))
        if kind == "point_add":
            a = [x + y for x, y in zip(a, _ints(_below(rng, case["n"], order, 8)))]
        return _points(curve, [2 * x for x in a] if kind == "point_dbl" else a)
    if kind in ("msm", "msm_ragged", "msm_bases"):
        a, k = _msm_inputs(case, seed)
        if kind == "msm_ragged":
            off = np.concatenate([[0], np.cumsum(_sizes(case))])
            return _points(curve, [_dot(a[i:j], k[i:j]) for i, j in zip(off[:-1], off[1:])])
        n = case["n"]
        return _points(curve, [_dot(a, k[v * n:(v + 1) * n]) for v in range(case.get("vectors", 1))])
    if case["n"] > 500:
        return None
    d, e, k, *_ = _ecdsa_inputs(case, seed)  # ECDSA signing with the given nonces
    d, e, k = ([int.from_bytes(bytes(x), "big") for x in v] for v in (d, e, k))
    r = [_times_g(curve, x)[0] % order for x in k]
    s = [pow(x, -1, order) * (h + y * z) % order for x, h, y, z in zip(k, e, r, d)]
    pub = [_times_g(curve, x) for x in d]

    def rows(vals):
        return np.frombuffer(b"".join(v.to_bytes(32, "big") for v in vals), dtype=np.uint8).reshape(-1, 32).copy()

    return {"r": rows(r), "s": rows(s), "pub": np.concatenate([rows([q[0] for q in pub]), rows([q[1] for q in pub])], axis=1)}
