"""CPU pins of the arithmetic of the residue products (csrc/rns.cu), from its
definitions: the moduli, the exactness of the FP32 steps (residues of 15-bit
pieces, quotients rounded by the add of 1.5 2^23, accumulators below 2^24) and
the limb sums that rebuild the integer."""
import math
import random

import numpy as np

MODULI = [256, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193]
P = math.prod(MODULI)
BETA = 58
MAGIC = np.float32(12582912.0)


def coef(l, j, scaled):
    p = MODULI[l]
    r = pow(2, 15 * j, p)
    if scaled:
        r = r * pow(P // p % p, -1, p) % p
    return r - p if r > p // 2 else r


def pieces(x):
    """Four 15-bit pieces of a signed integer, the top one signed."""
    return [x & 0x7FFF, (x >> 15) & 0x7FFF, (x >> 30) & 0x7FFF, x >> 45]


def residue(t, p):
    """t - p rint(t / p) in FP32, the quotient from one multiply-add (exact product, one rounding)."""
    inv = np.float32(1.0) / np.float32(p)
    q = np.float32(np.float64(t) * np.float64(inv) + np.float64(MAGIC)) - MAGIC
    return int(t) - p * int(q)


def test_moduli_and_bounds():
    assert all(math.gcd(a, b) == 1 for i, a in enumerate(MODULI) for b in MODULI[:i])
    assert 2 ** 117 <= P < 2 ** 118
    # operands of norm at most 2^58 give integers of at most 2^116, and their multiple of P is found by rounding
    assert 2 ** (2 * BETA) * (1 + 2 ** -20) < P / 2 * 0.8
    # 480 complex products of residues of magnitude 128, from a carried residue
    assert 2 * 480 * 128 * 128 + 128 < 2 ** 24
    for l in range(len(MODULI)):
        for scaled in (False, True):
            c = [abs(coef(l, j, scaled)) for j in range(4)]
            assert max(c) <= 128
            assert (sum(c[:3]) * 0x7FFF + c[3] * 2 ** 13) < 2 ** 24  # the piece sum is exact in FP32


def test_residues_of_pieces():
    rng = random.Random(1)
    xs = [0, 1, -1, 2 ** BETA, -2 ** BETA, 2 ** BETA - 1, 1 - 2 ** BETA]
    xs += [rng.randint(-2 ** BETA, 2 ** BETA) >> rng.randint(0, 58) for _ in range(400)]
    for x in xs:
        pc = pieces(x)
        assert sum(v << (15 * j) for j, v in enumerate(pc)) == x and abs(pc[3]) <= 2 ** 13
        for l, p in enumerate(MODULI):
            for scaled in (False, True):
                t = sum(coef(l, j, scaled) * v for j, v in enumerate(pc))
                assert abs(t) < 2 ** 24
                r = residue(t, p)
                want = x * (pow(P // p % p, -1, p) if scaled else 1)
                assert (r - want) % p == 0 and abs(r) <= 128
                assert int(np.array([r], np.float32).view(np.uint32)[0]) & 0xFFFF == 0  # exact in bfloat16


def test_reduction_of_accumulators():
    rng = random.Random(2)
    vals = [0, 2 ** 24, -2 ** 24] + [rng.randint(-2 ** 24, 2 ** 24) for _ in range(1000)]
    for p in MODULI:
        # the largest accumulators, where the quotient's error is largest, all at once
        a = np.concatenate([np.arange(-2 ** 24, -2 ** 24 + 2 ** 20), np.arange(2 ** 24 - 2 ** 20, 2 ** 24 + 1)]).astype(np.float64)
        q = (a * np.float64(np.float32(1) / np.float32(p)) + np.float64(MAGIC)).astype(np.float32) - MAGIC
        assert np.abs(a - p * q.astype(np.float64)).max() <= (127 if p < 256 else 128)
        for t in vals:
            r = residue(t, p)
            assert (r - t) % p == 0
            assert abs(r) <= (127 if p < 256 else 128)
            # the stored byte r + 128 stands for r (or, for p = 256, for an equal residue)
            assert (((r + 128) & 0xFF) - 128 - t) % p == 0


def limbs(v):
    return [v & 0xFFFFF, (v >> 20) & 0xFFFFFFFF, (v >> 52) & 0xFFFFFFFF, v >> 84]


def test_reconstruction_from_bytes():
    w = [limbs(P // p) for p in MODULI]
    bias = limbs(2 * P - 128 * sum(P // p for p in MODULI) % P)
    pl = limbs(P)
    assert 255 * sum(x[0] for x in w) < 2 ** 32  # the lowest limb's sum stays in 32 bits
    assert all(255 * sum(x[j] for x in w) + 2 ** 36 < 2 ** 63 for j in range(4))
    pinv = np.float32(np.float32(2.0 ** 84 / P) * np.float32(256.0))
    rng = random.Random(3)
    top = 2 ** (2 * BETA)
    xs = [0, 1, -1, top - 1, 1 - top, 2 ** 84, -2 ** 84, 2 ** 52, -2 ** 52, 2 ** 20, -2 ** 20]
    xs += [rng.randint(1 - top, top - 1) >> rng.randint(0, 116) for _ in range(2000)]
    for x in xs:
        u = []
        for p in MODULI:
            c = x * pow(P // p % p, -1, p) % p
            r = c - p if c > p // 2 else c
            u.append((r + 128) & 0xFF)
        a = [sum(q * x_[j] for q, x_ in zip(u, w)) + bias[j] for j in range(4)]
        assert a[3] >> 8 < 2 ** 32
        k = int(np.rint(np.float32(a[3] >> 8) * pinv))
        assert 0 <= k <= 22 and k * pl[0] < 2 ** 32
        s0 = a[0] - k * pl[0]
        s1 = a[1] - k * pl[1] + (s0 >> 20)
        s2 = a[2] - k * pl[2] + (s1 >> 32)
        s3 = a[3] - k * pl[3] + (s2 >> 32)
        assert (s3 << 84) + ((s2 & 0xFFFFFFFF) << 52) + ((s1 & 0xFFFFFFFF) << 20) + (s0 & 0xFFFFF) == x
        # the magnitude by inverting the words, with carries
        neg = s3 < 0
        low = ((s1 & 0xFFFFFFFF) << 20) | (s0 & 0xFFFFF)
        low = (low ^ (2 ** 52 - 1 if neg else 0)) + neg
        mid = ((s2 & 0xFFFFFFFF) ^ (0xFFFFFFFF if neg else 0)) + (low >> 52)
        A = (((s3 & 0xFFFFFFFF) ^ (0xFFFFFFFF if neg else 0)) + (mid >> 32)) & 0xFFFFFFFF
        low &= 2 ** 52 - 1
        assert (A << 84) + ((mid & 0xFFFFFFFF) << 52) + low == abs(x)
