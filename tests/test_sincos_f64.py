"""The FP64 sincos of the kernels (sincos2pi in bf_device.cuh): its table holds the correctly
rounded cosines and sines, and the steps evaluated in NumPy stay within 4e-16 of the exact
values.  Bound: the table entry and the joining sum round to half an ulp each (1.1e-16 + 1.1e-16),
the two products and the polynomials, at most 2 pi / 1024, add below 1e-17, the polynomials'
truncation 1e-17; products rounded twice where the kernels use FMAs add 1e-18."""
import decimal
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_4650_gb300", "csrc")
decimal.getcontext().prec = 50
TWO_PI = 2 * decimal.Decimal("3.14159265358979323846264338327950288419716939937510582")


def _exact(v):
    """cos and sin of 2 pi v by their series, 40 digits (|v| <= 1/2)."""
    x = TWO_PI * v
    c, s, term, n = decimal.Decimal(0), decimal.Decimal(0), decimal.Decimal(1), 0
    while abs(term) > decimal.Decimal("1e-42"):
        if n % 2 == 0:
            c += term if n % 4 == 0 else -term
        else:
            s += term if n % 4 == 1 else -term
        n += 1
        term = term * x / n
    return c, s


def _octant():
    src = open(os.path.join(CSRC, "bf_sctab.h")).read()
    body = src[src.index("kOctant[65]"):]
    rows = re.findall(r"\{(-?0x[0-9a-fp.+-]+), (-?0x[0-9a-fp.+-]+)\}", body[:body.index("};")])
    return np.array([[float.fromhex(a), float.fromhex(b)] for a, b in rows])


def _circle(o):
    k = np.arange(512)
    r = k % 128
    m = np.where(r <= 64, r, 128 - r)
    c = np.where(r <= 64, o[m, 0], o[m, 1])
    s = np.where(r <= 64, o[m, 1], o[m, 0])
    quad = k // 128
    return (np.choose(quad, [c, -s, -c, s]), np.choose(quad, [s, c, -s, -c]))


def test_table_is_correctly_rounded():
    o = _octant()
    assert o.shape == (65, 2)
    for k in range(65):
        c, s = _exact(decimal.Decimal(k) / 512)
        assert o[k, 0] == float(c) and o[k, 1] == float(s), k


def test_steps_against_exact_values():
    src = open(os.path.join(CSRC, "bf_device.cuh")).read()
    body = src[src.index("void sincos2pi(double v"):]
    body = body[:body.index("\n}")]
    s2, s1, s0 = (float(x) for x in re.search(r"sn = r \* fma\(u, fma\(u, ([-0-9.]+), ([-0-9.]+)\), ([-0-9.]+)\)", body).groups())
    c2, c1 = (float(x) for x in re.search(r"cm = u \* fma\(u, ([-0-9.]+), ([-0-9.]+)\)", body).groups())
    C, S = _circle(_octant())
    rng = np.random.default_rng(3)
    edge = (np.arange(-40, 41) + 0.5) / 512          # half way between table entries
    v = np.concatenate([rng.uniform(-0.5, 0.5, 1500), edge, np.nextafter(edge, 1), [0.0, 0.125, -0.25, 0.5]])
    M = 6755399441055744.0
    t = v * 512.0 + M
    k = ((t - M).astype(np.int64)) & 511
    r = v - (t - M) / 512.0
    u = r * r
    sn = r * (u * (u * s2 + s1) + s0)
    cm = u * (u * c2 + c1)
    c = C[k] + (C[k] * cm - S[k] * sn)
    s = S[k] + (S[k] * cm + C[k] * sn)
    for i, x in enumerate(v):
        ec, es = _exact(decimal.Decimal(float(x)))
        assert abs(decimal.Decimal(float(c[i])) - ec) <= decimal.Decimal("4e-16"), x
        assert abs(decimal.Decimal(float(s[i])) - es) <= decimal.Decimal("4e-16"), x
