"""CPU model of the FP64-class products through residues (csrc/crt.cu): moduli, residue ranges, exact chunk sums and
the reconstruction, in Python integers."""
import math
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = open(os.path.join(ROOT, "paper_2205_02491_gb300", "csrc", "crt.cu")).read()
MODULI = [int(x) for x in re.search(r"#define CRT_MODULI \{([^}]*)\}", SRC).group(1).split(",")]
M = math.prod(MODULI)


def test_moduli_are_coprime_and_wide_enough():
    assert len(MODULI) == 16 and max(MODULI) <= 256
    for i, a in enumerate(MODULI):
        for b in MODULI[i + 1:]:
            assert math.gcd(a, b) == 1
    # |C| <= 2^62 2^62 lies inside (-M/2, M/2), well away from its ends (the FP32 quotient's slack)
    assert 2 ** 124 < 0.33 * M and 2 ** 125 <= M < 2 ** 126
    # 1024 products of residues are an exact FP32 sum
    assert 1024 * 128 * 128 <= 2 ** 24


def sym(x, m):
    r = x % m
    return r - m if r > m // 2 else r


def residue(x, m):
    """The kernel's residue of a 63-bit integer: 21-bit limbs, 32-bit sums, quotient by multiply and shift."""
    x0, x1, x2 = x & 0x1fffff, (x >> 21) & 0x1fffff, x >> 42
    t = x0 + x1 * sym(2 ** 21, m) + x2 * sym(2 ** 42, m)
    assert -2 ** 30 < t < 2 ** 30
    inv = (2 ** 38 + m // 2) // m
    assert inv < 2 ** 31
    q = (t * inv + 2 ** 37) >> 38
    return t - q * m


@pytest.mark.parametrize("m", MODULI)
def test_residues_stay_in_bf16_range(m):
    g = np.random.default_rng(m)
    xs = [0, 1, -1, 2 ** 62, -2 ** 62, 2 ** 62 - 1, m // 2, m // 2 + 1, -(m // 2)]
    xs += [int(v) for v in g.integers(-2 ** 62, 2 ** 62, size=4000)]
    xs += [int(v) * m + m // 2 for v in g.integers(-2 ** 52, 2 ** 52, size=1000)]
    for x in xs:
        r = residue(x, m)
        assert abs(r) <= 128 and (r - x) % m == 0


def test_products_come_back_exactly():
    """Three residue products per modulus give the exact complex integer product at any magnitude up to the bound."""
    g = np.random.default_rng(5)
    w = []
    for m in MODULI:
        Mi = M // m
        w.append(Mi * pow(Mi, -1, m))
    for bits in (1, 20, 55, 58):
        K = 7
        top = 2 ** bits
        xr, xi, yr, yi = ([int(v) for v in g.integers(-top, top + 1, size=K)] for _ in range(4))
        cr = sum(a * c - b * d for a, b, c, d in zip(xr, xi, yr, yi))
        ci = sum(a * d + b * c for a, b, c, d in zip(xr, xi, yr, yi))
        sr = si = 0
        for m, wi in zip(MODULI, w):
            p1 = sum(residue(a, m) * residue(c, m) for a, c in zip(xr, yr))
            p2 = sum(residue(b, m) * residue(d, m) for b, d in zip(xi, yi))
            p3 = sum(residue(a + b, m) * residue(c + d, m) for a, b, c, d in zip(xr, xi, yr, yi))
            p1, p2, p3 = (sym(p, m) for p in (p1, p2, p3))
            sr += (p1 - p2 + 512) * wi
            si += (p3 - p1 - p2 + 512) * wi
            assert p1 - p2 + 512 > 0 and p3 - p1 - p2 + 512 > 0
        off = (-512 * sum(w)) % M
        for s, c in ((sr, cr), (si, ci)):
            t = s + off
            q = int(np.rint(np.float32((t >> 112) & 0xffffffff) * np.float32(2.0 ** 48 / float(M >> 64))))
            assert t >> 144 == 0
            assert t - q * M == c
