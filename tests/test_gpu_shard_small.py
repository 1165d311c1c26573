"""Sharded applies of the smallest grids, where a rank holds as little as one pair of a pass: the
parts of all ranks, computed one after another on one GPU, sum to the oracle's result.  One pair
of odd q is where the shared-memory arrays of a CTA end off a 16-byte boundary.

Tolerances (relative l2) as in test_gpu_routes.py: FP64 1e-11, mixed 1e-5; a result that cancels
to nothing is held against the input."""
import numpy as np
import pytest

import oracle
from paper_1305_4650_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-11, "mixed": 1e-5}


@pytest.fixture(scope="module")
def bf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_4650_gb300 import build, bf as bfmod
    build.build()
    return bfmod


def check(bf, spec, nrhs, precision, sg):
    import torch
    dt = np.complex128 if precision == "fp64" else np.complex64
    g = wl.source_values(spec, nrhs, dt, seed=90 + spec.q)
    x = torch.from_numpy(g).cuda()
    plan = bf.Plan.from_spec(spec, max_nrhs=nrhs, precision=precision)
    out = sum(plan.apply_shard(x, sg, r).cpu().numpy().reshape(nrhs, -1).astype(np.complex128) for r in range(1 << sg))
    plan.close()
    P = oracle.Problem(**spec.oracle_kwargs())
    for j in range(nrhs):
        ref, inp = oracle.butterfly(P, g[j].astype(np.complex128)), np.linalg.norm(g[j])
        size = np.linalg.norm(ref)
        assert np.linalg.norm(out[j] - ref) <= TOL[precision] * (size if size > 1e-12 * inp else inp), j


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("phase", ["genradon", "dot"])
@pytest.mark.parametrize("off", [0.0, 0.5])
@pytest.mark.parametrize("L,q,m,sg", [(1, 3, None, 2), (1, 5, None, 2), (1, 5, None, 1), (1, 4, None, 2), (2, 5, 0, 2),
                                      (2, 3, 1, 2), (2, 2, None, 2)])
def test_one_right_hand_side(bf, L, q, m, sg, off, phase, precision):
    base = wl.genradon2d(L, precision)
    check(bf, base.with_(q=q, m=m, phase=phase, tgt_off=off, src_off=off), 1, precision, sg)


@pytest.mark.parametrize("nrhs", [2, 3, 17])
@pytest.mark.parametrize("off,node_kind", [(0.0, 0), (0.5, 0), (0.25, 1)])
@pytest.mark.parametrize("L,q,m,sg", [(1, 3, None, 2), (1, 5, None, 2), (1, 4, None, 2), (2, 5, 0, 2), (2, 3, None, 1)])
def test_several_right_hand_sides(bf, L, q, m, sg, off, node_kind, nrhs):
    """One pair of odd q and an odd number of right-hand sides: the weights of the first step are an
    odd number of complex numbers, every one of them set."""
    spec = wl.genradon2d(L).with_(q=q, m=m, phase="hypradon" if nrhs == 2 else "genradon", tgt_off=off, src_off=off, node_kind=node_kind)
    if spec.phase == "hypradon":
        spec = spec.with_(x_lo=(1.0, 0.0, 0.0), y_lo=(1.0, 0.0, 0.0), y_w=(1.0, 1.0, 1.0), scale=float(1 << L))
    check(bf, spec, nrhs, "mixed", sg)
