"""Plans whose roots are large and reach small values keep the rounding error of the sums under the
root (wide_root, csrc/bf_host.h): the phases, and every kind of apply, at roots up to the
accepted bound |Phi| < 2^21.

Tolerances as in test_gpu_selfcheck.py (3e-7 cycles) and test_gpu_routes.py (relative l2, d = 2 1e-5,
d = 3 and the split-precision switches 1e-4).  One source near p = 0 sees small roots only: on one
common grid its phases were off by up to 6e-5 cycles."""
import numpy as np
import pytest

import oracle
from paper_1305_4650_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
BIG = 70000.0                        # N = 16: |Phi| to 1.9e6 cycles, roots to 7.9e5


@pytest.fixture(scope="module")
def bf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_4650_gb300 import build, bf as bfmod
    build.build()
    return bfmod


def near_zero(spec, nrhs, seed=3):
    """Sources at p = 0 and its neighbours only."""
    rng, n = np.random.default_rng(seed), spec.N
    g = np.zeros((nrhs,) + (n,) * spec.d, np.complex64)
    box = (slice(None),) + (slice(n // 2 - 1, n // 2 + 2),) * spec.d
    g[box] = rng.standard_normal(g[box].shape) + 1j * rng.standard_normal(g[box].shape)
    return g.reshape(nrhs, -1)


def errors(spec, got, g, adjoint=False):
    P = oracle.Problem(**spec.oracle_kwargs())
    ref = oracle.butterfly_adjoint if adjoint else oracle.butterfly
    out = []
    for a, b in zip(np.asarray(got).reshape(len(g), -1), g):
        r = ref(P, b.astype(np.complex128))
        out.append(np.linalg.norm(a - r) / np.linalg.norm(r))
    return max(out)


@pytest.mark.parametrize("precision", ["mixed", "mixed_sfu"])
@pytest.mark.parametrize("spec", [wl.genradon2d(11), wl.genradon2d(14), wl.genradon2d(10).with_(scale=30.0),
                                  wl.genradon2d(10).with_(scale=-1000.0), wl.genradon3d(5).with_(scale=20000.0),
                                  wl.hypradon(9).with_(scale=3e5, y_lo=(0.0, 0.0, 0.0))],
                         ids=["N2048", "N16384", "root2e4", "root7e5", "d3", "hypradon"])
def test_phases_against_fp64(bf, spec, precision):
    plan = bf.Plan.from_spec(spec, precision=precision) if spec.L < 14 else bf.Plan.from_spec(spec.with_(q=2), precision=precision)
    err = plan.selfcheck_phase(1 << 20)
    plan.close()
    assert err < 3e-7, err


@pytest.mark.parametrize("precision,nrhs,tables,tol", [("mixed", 1, False, 1e-5), ("mixed", 3, False, 1e-5), ("mixed", 1, True, 1e-5),
                                                       ("mixed", 3, True, 1e-5), ("mixed_sfu", 1, False, 1e-5),
                                                       ("mixed_sfu", 2, False, 1e-5), ("bf16x3", 3, False, 1e-4), ("tf32x3", 3, False, 1e-4)])
@pytest.mark.parametrize("q,node_kind", [(5, 0), (4, 1)])
def test_applies(bf, q, node_kind, precision, nrhs, tables, tol):
    import torch
    spec = wl.genradon2d(4).with_(q=q, node_kind=node_kind, scale=BIG)
    g = near_zero(spec, nrhs)
    plan = bf.Plan.from_spec(spec, max_nrhs=nrhs, precision=precision, phase_tables=tables)
    x = torch.from_numpy(g).cuda()
    assert errors(spec, plan.apply(x).cpu().numpy(), g) <= tol
    assert errors(spec, plan.apply_adjoint(x).cpu().numpy(), g, adjoint=True) <= 1e-5
    plan.close()


def test_space(bf):
    import torch
    spec = wl.genradon3d(3).with_(scale=60000.0)
    g = near_zero(spec, 2)
    plan = bf.Plan.from_spec(spec, max_nrhs=2)
    x = torch.from_numpy(g).cuda()
    assert errors(spec, plan.apply(x).cpu().numpy(), g) <= 1e-4
    assert errors(spec, plan.apply_adjoint(x).cpu().numpy(), g, adjoint=True) <= 1e-4
    plan.close()


def test_hyperbolic_from_zero_points_and_no_allocation(bf):
    import torch
    spec = wl.hypradon(4).with_(scale=2e5, y_lo=(0.0, 0.0, 0.0))
    rng = np.random.default_rng(5)
    y, x = rng.random((60, 2)) * 0.02, np.array([1.0, 0.0]) + rng.random((50, 2))
    g = (rng.standard_normal((3, 60)) + 1j * rng.standard_normal((3, 60))).astype(np.complex64)
    plan = bf.Plan.from_spec(spec, max_nrhs=3, sources=y, targets=x)
    out = plan.apply(torch.from_numpy(g).cuda()).cpu().numpy()
    plan.close()
    ref = oracle.butterfly_points(oracle.Problem(**spec.oracle_kwargs()), y, g.astype(np.complex128), x)
    assert (np.linalg.norm(out - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= 1e-5
    h = np.zeros((1, spec.npts), np.complex64)
    h[0, :3] = 1.0
    f = torch.empty(1, spec.npts, dtype=torch.complex64, device="cuda")
    x_lo, x_w, y_lo, y_w = spec.domain()
    bf.apply_noalloc(2, spec.N, spec.q, spec.phase, torch.from_numpy(h).cuda(), f, scale=spec.scale, x_lo=x_lo, x_w=x_w, y_lo=y_lo,
                     y_w=y_w, switch_level=spec.switch_level)
    assert errors(spec, f.cpu().numpy(), h) <= 1e-5


def test_persistent_batch_of_both_forms(bf):
    """A plan on the grid and one with exact sums in one launch: the first one's results do not change."""
    import torch
    specs = [wl.genradon2d(5), wl.genradon2d(4).with_(scale=BIG), wl.genradon2d(5).with_(scale=2.0)]
    nr = [2, 3, 1]
    plans = [bf.Plan.from_spec(s, max_nrhs=n) for s, n in zip(specs, nr)]
    gs = [near_zero(s, n) for s, n in zip(specs, nr)]
    gs = [g if g.shape[0] > 1 else wl.source_values(specs[2], 1, np.complex64, seed=1) for g in gs]
    xs = [torch.from_numpy(g).cuda() for g in gs]
    fs = [torch.empty_like(x) for x in xs]
    batch = bf.Batch(plans, nr)
    batch.apply(xs, fs)
    for s, g, f in zip(specs, gs, fs):
        assert errors(s, f.cpu().numpy(), g) <= 1e-5
    assert torch.equal(fs[0], plans[0].apply(xs[0]))
    assert not batch.status()
    batch.close()
    for p in plans:
        p.close()
