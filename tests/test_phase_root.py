"""The sums of squares under a root in the mixed precisions: which plans add the terms on one grid
and which keep the rounding error of the sum (wide_root, sqrt_grid in csrc/bf_host.h, evaluated on
the host), and the error of both forms in NumPy float32, operation by operation as the kernels
have them, over all roots of a plan's domain.

Bound, in cycles: one FP32 rounding of the reduced phase, at most 1/2, and of each of the three
steps before it (3e-8 each at most, 1.2e-7), and the 6e-8 that the rule allows the grid.  At roots of 1e6
cycles the grid alone would be off by 4e-5."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include "bf_host.h"
int main()
{
    bf_params p;
    int d, kind, prec;
    double s, xlo, xw, ylo, yw;
    while (std::scanf("%d %d %d %lf %lf %lf %lf %lf", &d, &kind, &prec, &s, &xlo, &xw, &ylo, &yw) == 8) {
        p = bf_params();
        for (int k = 0; k < 3; ++k) { p.x_lo[k] = k ? 0.0 : xlo; p.x_w[k] = xw; p.y_lo[k] = ylo; p.y_w[k] = yw; }
        if (kind == BF_PHASE_HYPRADON) p.y_lo[1] = 0.0;
        p.phase_scale = s;
        p.precision = (bf_precision)prec;
        double lin, root;
        bfl::phase_bounds(d, kind, &p, &lin, &root);
        std::printf("%d %.9g %.17g %.17g\n", (int)bfl::wide_root(d, kind, &p), bfl::sqrt_grid(d, kind, &p), root,
                    bfl::root_floor(d, kind, &p));
    }
}
"""
FP64, MIXED, SFU, BF16 = 0, 1, 2, 3
DOT, GEN, HYP, SEP = 0, 1, 2, 3
# (d, kind, precision, scale, first target coordinate's start, widths, source start and width), wide?
CASES = [((2, GEN, MIXED, 1.0, 0.0, 1.0, -512.0, 1024.0), False),     # N = 1024: roots to 724
         ((2, GEN, SFU, 1.0, 0.0, 1.0, -1024.0, 2048.0), True),
         ((2, GEN, BF16, -70000.0, 0.0, 1.0, -8.0, 16.0), True),
         ((2, GEN, MIXED, 40.0, 0.0, 1.0, 512.0, 1024.0), False),      # far from the origin
         ((2, GEN, FP64, 70000.0, 0.0, 1.0, -8.0, 16.0), False),
         ((3, GEN, MIXED, 1.0, 0.0, 1.0, -32.0, 64.0), False),
         ((3, GEN, MIXED, 2000.0, 0.0, 1.0, -2.0, 4.0), True),
         ((2, HYP, MIXED, 512.0, 1.0, 1.0, 1.0, 1.0), False),          # tau, w in [1, 2)
         ((2, HYP, MIXED, 32768.0, 1.0, 1.0, 1.0, 1.0), False),
         ((2, HYP, MIXED, 32768.0, 1.0, 1.0, 0.0, 1.0), True),         # tau from 0
         ((2, HYP, MIXED, 32768.0, 0.0, 1.0, 1.0, 1.0), True),         # w from 0
         ((2, DOT, MIXED, 1000.0, 0.0, 1.0, -512.0, 1024.0), False),
         ((2, SEP, MIXED, 1.0, 0.0, 1.0, -512.0, 1024.0), False)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    from paper_1305_4650_gb300 import build
    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    tmp = tmp_path_factory.mktemp("root")
    (tmp / "root.cu").write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                    *build.ARCH, str(tmp / "root.cu"), "-o", str(tmp / "root")], check=True)
    text = "\n".join(" ".join(repr(v) for v in c) for c, _ in CASES)
    out = subprocess.run([str(tmp / "root")], input=text, capture_output=True, text=True, check=True).stdout
    return [tuple(float(v) for v in line.split()) for line in out.splitlines()]


f32, f64, wide_t = np.float32, np.float64, np.longdouble


def _split(x):
    h = x.astype(f32)
    return h, (x - h.astype(f64)).astype(f32)


def _fma(a, b, c):
    return (a.astype(wide_t) * b.astype(wide_t) + c.astype(wide_t)).astype(f32)


def _mul(x, y):
    p = x[0] * y[0]
    return p, _fma(x[1], y[0], _fma(x[0], y[1], _fma(x[0], y[0], -p)))


def root_error(mg, wide, big, lo, n=40000):
    """Largest error of the reduced root, roots spread over [lo, big], d = 2."""
    rng, worst = np.random.default_rng(1), 0.0
    for sig in np.geomspace(max(lo, big * 2.0 ** -16) * 1.2, big, 24):
        s = sig * rng.uniform(1 / 1.2, 1.0, n)
        th = rng.uniform(0, np.pi / 2, n)
        exact, H, Lo = 0, [], []
        for k, c in enumerate((np.cos(th), np.sin(th))):
            a = big * rng.uniform(1 / 3, 1, n)
            A = _mul(_split(a), _split(a))
            Y = _split((s * c / a) ** 2)
            p = _mul(A, Y)
            exact = exact + (A[0].astype(wide_t) + A[1]) * (Y[0].astype(wide_t) + Y[1])
            h = (p[0] + f32(mg)) - f32(mg)
            H.append(h)
            Lo.append(((p[0] - h) + p[1]) + f32(1e-30 if k == 0 else 0))
        h, l = H[0] + H[1], Lo[0] + Lo[1]
        if wide:
            b = h - H[0]
            l = l + ((H[0] - (h - b)) + (H[1] - b))
        M = f32(12582912)
        q = h + l
        r = (1 / np.sqrt(q.astype(f64))).astype(f32)
        x = q * r
        w = x - ((x + M) - M)
        e = _fma(f32(0.5) * np.ones_like(r), (_fma(-x, x, h) + l) * r, w).astype(wide_t) - np.sqrt(exact)
        worst = max(worst, float(np.abs(e - np.rint(e)).max()))
    return worst


def test_rule(rule):
    assert [bool(r[0]) for r in rule] == [w for _, w in CASES]
    for (_, mg, big, _), (case, wide) in zip(rule, CASES):
        if case[2] != FP64:
            assert (mg == 0.0) == wide


@pytest.mark.parametrize("i", [i for i, (c, _) in enumerate(CASES) if c[0] == 2 and c[1] in (GEN, HYP) and c[2] != FP64])
def test_both_forms_hold_the_bound(rule, i):
    wide, mg, big, lo = rule[i]
    assert root_error(mg, bool(wide), big, lo) <= 1.2e-7 + 6e-8


def test_exact_sums_change_nothing_on_a_grid(rule):
    """The kernels with exact sums serve plans on the grid too (batches): every error term is zero."""
    _, mg, big, lo = rule[0]
    assert root_error(mg, True, big, lo) == root_error(mg, False, big, lo)
    assert root_error(1.5 * 2.0 ** 43, False, 2.0 ** 20, 0.0) > 1e-5       # the grid where it does not serve
