"""The passes that a plan chooses by sizes, nodes, offsets and number of right-hand sides,
forward and adjoint, against the FP64 CPU oracle: corner grids (points at offset 0 with
Lobatto nodes of odd q, whose end levels use one or four nodes of a box) beside every other
combination of offsets and nodes, even and odd q, switch levels that leave the end levels to
either kind of pass, one and several right-hand sides up to one more than a CTA holds, and
one, two or three fused levels.

Tolerances (relative l2, as in test_gpu_parity.py): FP64 1e-11; mixed 1e-5 at d = 2, 1e-4 at
d = 3 (a few 1e-7 per level over at most 2 L + 2 steps; the phases are good to 2^-44)."""
import numpy as np
import pytest

import oracle
from paper_1305_4650_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {("fp64", 2): 1e-11, ("mixed", 2): 1e-5, ("fp64", 3): 1e-11, ("mixed", 3): 1e-4}


@pytest.fixture(scope="module")
def bf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_4650_gb300 import build, bf as bfmod
    build.build()
    return bfmod


def spec_of(d, L, q, phase, **kw):
    base = dict(x_lo=(0.0,) * 3, x_w=(1.0,) * 3)
    if phase == "hypradon":
        base = dict(x_lo=(1.0, 0.0, 0.0), y_lo=(1.0, 0.0, 0.0), y_w=(1.0, 1.0, 1.0), scale=float(1 << L))
    base.update(kw)
    return wl.Spec(f"t_{d}_{L}_{q}_{phase}", d, L, q, phase, **base)


def check(bf, spec, nrhs, precision, fuse=0):
    """Forward and adjoint of one plan, every right-hand side against the oracle's."""
    import torch
    dt = np.complex128 if precision == "fp64" else np.complex64
    P = oracle.Problem(**spec.oracle_kwargs())
    two = wl.source_values(spec, 2, dt, seed=7 + spec.L)   # right-hand sides: mixes of two
    mix = np.exp(1j * np.arange(nrhs))[:, None]
    amp = (1.0 + np.arange(nrhs) % 3)[:, None]
    v = (two[:1] + (amp * mix) * two[1:]).astype(dt)
    plan = bf.Plan.from_spec(spec, max_nrhs=nrhs, precision=precision, fuse_levels=fuse)
    x = torch.from_numpy(np.ascontiguousarray(v)).cuda()
    for run, ref in ((plan.apply, oracle.butterfly), (plan.apply_adjoint, oracle.butterfly_adjoint)):
        b = ref(P, two.astype(np.complex128))
        want = b[:1] + (amp * mix) * b[1:]
        out = run(x)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        # a result that cancels to nothing (d = 3, L = 1, q = 2 with sources in the middle of their
        # boxes: 1.6e-16 of the input in the oracle) is held against the input instead
        size, inp = np.linalg.norm(want, axis=1), np.linalg.norm(v, axis=1)
        err = np.linalg.norm(got - want, axis=1) / np.where(size > 1e-12 * inp, size, inp)
        assert err.max() <= TOL[(precision, spec.d)], (run.__name__, err)
    plan.close()


GRIDS = [
    # corner grids and their neighbours: (L, q, phase, extra, nrhs, fuse)
    (1, 5, "genradon", {}, 1, 0),
    (1, 3, "hypradon", {}, 2, 0),
    (2, 5, "hypradon", {"m": 0}, 3, 0),
    (2, 5, "hypradon", {"m": 1}, 3, 0),
    (3, 5, "genradon", {"m": 1}, 1, 1),
    (3, 5, "genradon", {"m": 2}, 17, 2),
    (4, 5, "dot", {"m": 3}, 1, 3),
    (4, 5, "hypradon", {}, 16, 0),
    (5, 3, "separable", {}, 2, 0),
    (5, 3, "genradon", {"m": 4}, 1, 0),
    (5, 5, "genradon", {"tgt_off": 0.5}, 1, 0),
    (5, 5, "genradon", {"src_off": 0.5}, 1, 0),
    (4, 5, "hypradon", {"tgt_off": 0.5}, 3, 0),
    (4, 5, "hypradon", {"src_off": 0.5}, 3, 0),
    (4, 5, "genradon", {"node_kind": 1}, 1, 0),
    (4, 5, "hypradon", {"node_kind": 1}, 3, 0),
    (6, 5, "genradon", {}, 1, 0),
    (8, 3, "genradon", {}, 1, 0),     # more CTAs than SMs
    (8, 3, "hypradon", {}, 2, 0),
]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", GRIDS, ids=[f"L{c[0]}q{c[1]}{c[2]}n{c[4]}k{c[5]}" + "".join(f"_{k}{v}" for k, v in c[3].items())
                                            for c in GRIDS])
def test_corner_grids_and_neighbours(bf, case, precision):
    L, q, phase, kw, nrhs, fuse = case
    check(bf, spec_of(2, L, q, phase, **kw), nrhs, precision, fuse)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("q", [2, 3, 4, 6, 8])
def test_every_q(bf, q, nrhs, precision):
    check(bf, spec_of(2, 4, q, "hypradon", tgt_off=0.25 if q == 6 else 0.0), nrhs, precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("off", [(0.0, 0.0), (0.5, 0.0), (0.0, 0.5)])
@pytest.mark.parametrize("L,q,m", [(1, 2, None), (2, 4, 0), (3, 3, 2), (3, 4, 1), (4, 2, 3)])
def test_leaf_nodes_3d(bf, L, q, m, off, precision):
    check(bf, spec_of(3, L, q, "genradon", m=m, tgt_off=off[0], src_off=off[1]), 2, precision)


@pytest.mark.parametrize("nrhs", [10, 16])
def test_multi_rhs_shared_memory_above_48k(bf, nrhs):
    """Dynamic shared memory just under 48 KB together with a kernel's static arrays."""
    check(bf, spec_of(2, 6, 6, "hypradon"), nrhs, "mixed")


@pytest.mark.parametrize("L,q,m,phase,nrhs,precision", [
    (3, 4, 0, "hypradon", 2, "mixed"), (4, 5, None, "genradon", 17, "mixed"), (5, 8, None, "hypradon", 3, "mixed"),
    (4, 5, 3, "dot", 3, "fp64"), (1, 3, None, "genradon", 2, "fp64")])
def test_points_with_several_right_hand_sides(bf, L, q, m, phase, nrhs, precision):
    """The merges of a plan for scattered points by the multi-RHS passes, none of whose end levels
    is a corner grid's."""
    import torch
    spec = spec_of(2, L, q, phase, m=m)
    rng = np.random.default_rng(L + q)
    x_lo, x_w, y_lo, y_w = spec.domain()
    y = np.asarray(y_lo[:2]) + rng.random((150, 2)) * np.asarray(y_w[:2])
    x = np.asarray(x_lo[:2]) + rng.random((120, 2)) * np.asarray(x_w[:2])
    dt = np.complex128 if precision == "fp64" else np.complex64
    g = (rng.standard_normal((nrhs, 150)) + 1j * rng.standard_normal((nrhs, 150))).astype(dt)
    plan = bf.Plan.from_spec(spec, max_nrhs=nrhs, precision=precision, sources=y, targets=x)
    out = plan.apply(torch.from_numpy(g).cuda()).cpu().numpy()
    plan.close()
    ref = oracle.butterfly_points(oracle.Problem(**spec.oracle_kwargs()), y, g.astype(np.complex128), x)
    err = np.linalg.norm(out - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= TOL[(precision, 2)], err
