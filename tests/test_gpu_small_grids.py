"""Launch shapes of small grids, forward and adjoint, against the FP64 CPU oracle: more threads than a
stage has items, the next stage's preparation on the threads that are left over, and the first level's
parts beside its geometry; grids of one CTA per SM and of more.

Tolerances (relative l2) as in test_gpu_routes.py: FP64 1e-11, mixed 1e-5."""
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


def spec_of(L, q, phase, off):
    s = wl.hypradon(L) if phase == "hypradon" else wl.genradon2d(L).with_(phase=phase)
    return s.with_(q=q, tgt_off=off, src_off=off)


def inputs(spec, nrhs, precision):
    dt = np.complex128 if precision == "fp64" else np.complex64
    two = wl.source_values(spec, 2, dt, seed=11 + spec.L)          # right-hand sides: mixes of two
    mix, amp = np.exp(1j * np.arange(nrhs))[:, None], (1.0 + np.arange(nrhs) % 3)[:, None]
    return two, amp * mix, (two[:1] + (amp * mix) * two[1:]).astype(dt)


def compare(bf, spec, nrhs, precision):
    """Forward and adjoint of one plan, every right-hand side against the oracle's."""
    import torch
    two, c, v = inputs(spec, nrhs, precision)
    P = oracle.Problem(**spec.oracle_kwargs())
    plan = bf.Plan.from_spec(spec, max_nrhs=nrhs, precision=precision)
    x = torch.from_numpy(v).cuda()
    for run, ref in ((plan.apply, oracle.butterfly), (plan.apply_adjoint, oracle.butterfly_adjoint)):
        b = ref(P, two.astype(np.complex128))
        want, got = b[:1] + c * b[1:], run(x).cpu().numpy()
        err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
        assert err.max() <= TOL[precision], (run.__name__, err)
    plan.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("L,q,phase,off", [(1, 3, "hypradon", 0.5), (2, 2, "dot", 0.5), (3, 6, "genradon", 0.5), (4, 8, "dot", 0.0),
                                           (5, 3, "hypradon", 0.5), (5, 4, "dot", 0.5), (5, 6, "genradon", 0.0), (6, 2, "hypradon", 0.0),
                                           (6, 5, "genradon", 0.5), (7, 4, "dot", 0.0), (7, 3, "genradon", 0.5)])
def test_one_right_hand_side(bf, L, q, phase, off, precision):
    compare(bf, spec_of(L, q, phase, off), 1, precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("L,q,phase,off,nrhs", [(5, 8, "hypradon", 0.0, 2), (5, 5, "genradon", 0.5, 2), (4, 8, "dot", 0.0, 3),
                                                (4, 5, "hypradon", 0.0, 5), (3, 6, "genradon", 0.5, 17), (5, 3, "hypradon", 0.5, 16),
                                                (2, 4, "dot", 0.5, 9), (1, 5, "genradon", 0.0, 33)])
def test_several_right_hand_sides(bf, L, q, phase, off, nrhs, precision):
    compare(bf, spec_of(L, q, phase, off), nrhs, precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_blocks_of_right_hand_sides_do_not_change_a_result(bf, precision):
    """N = 16 in FP64: 16 right-hand sides in blocks of two, five one by one."""
    import torch
    spec = spec_of(4, 5, "hypradon", 0.5)
    _, _, v = inputs(spec, 16, precision)
    plan = bf.Plan.from_spec(spec, max_nrhs=16, precision=precision)
    x = torch.from_numpy(v).cuda()
    f, g = plan.apply(x), plan.apply_adjoint(x)
    assert torch.equal(plan.apply(x[3:8]), f[3:8])
    assert torch.equal(plan.apply_adjoint(x[3:8]), g[3:8])
    plan.close()


@pytest.mark.parametrize("L,q,phase", [(6, 3, "hypradon"), (6, 4, "genradon"), (6, 6, "hypradon"), (7, 2, "dot"), (5, 8, "dot")])
def test_two_right_hand_sides_of_the_adjoint_run_as_one_each(bf, L, q, phase):
    """Where the single-RHS passes fill the SMs once, two right-hand sides give the bits of one at a time."""
    import torch
    spec = spec_of(L, q, phase, 0.5)
    _, _, v = inputs(spec, 2, "mixed")
    plan = bf.Plan.from_spec(spec, max_nrhs=2)
    x = torch.from_numpy(v).cuda()
    both = plan.apply_adjoint(x)
    assert all(torch.equal(both[j], plan.apply_adjoint(x[j:j + 1])[0]) for j in range(2))
    plan.close()
    compare(bf, spec, 2, "mixed")
