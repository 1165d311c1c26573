"""Cases that time the butterfly's public entry points, and their results in 64 bits.

A case is a dict of plain values.  ``call`` says which entry point it goes through:

* ``apply``     ``Plan.apply`` (grid plans; with ``tables`` a plan that keeps its phases)
* ``gradient``  ``autograd.butterfly`` and its backward: one forward and one adjoint apply
* ``cgls``      ``autograd.cgls``: ``iters`` iterations of one forward and one adjoint apply
* ``points``    ``Plan.apply`` of a plan for scattered sources and targets
* ``batch``     ``bf.apply_batched`` over several plans of uneven size

``exact`` computes the same approximate operator (the Chebyshev-interpolation butterfly,
every level of it) with plain torch operations in 64 bits, from the formulas alone.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1305_4650_gb300 import autograd, bf, workloads

# Default node counts of the configurations: 5 per dimension in the plane, 4 in space.
BASE = {"call": "apply", "d": 2, "L": 10, "q": 5, "phase": "genradon", "precision": "mixed", "nrhs": 1}


def _case(**kw) -> dict:
    return {**BASE, **kw}


def listed() -> list[dict]:
    return [
        # the Fourier check of the method in double precision: a small transform, called often
        _case(name="fourier_n64_fp64", L=6, phase="dot", precision="fp64"),
        # a small single transform: few CTAs, so launches and latency count
        _case(name="genradon2d_n128", L=7),
        # the headline problem: one generalized Radon transform of 2^20 points
        _case(name="genradon2d_n1024", L=10),
        # the same operator applied many times, phases kept by the plan
        _case(name="genradon2d_n512_tables", L=9, tables=True),
        # the volume problem
        _case(name="genradon3d_n64", d=3, L=6, q=4),
        # double precision with a few right-hand sides: the accuracy reference of a batch
        _case(name="hypradon_n128_fp64_4rhs", L=7, phase="hypradon", precision="fp64", nrhs=4),
        # a full block of right-hand sides of one hyperbolic Radon operator
        _case(name="hypradon_n512_16rhs", L=9, phase="hypradon", nrhs=16),
        # the same with the switch on the tensor cores
        _case(name="hypradon_n512_16rhs_bf16x3", L=9, phase="hypradon", nrhs=16, precision="bf16x3"),
        # one step of an inversion with several gathers: value and gradient
        _case(name="hypradon_n256_7rhs_gradient", call="gradient", L=8, phase="hypradon", nrhs=7),
        # many independent transforms of uneven size and right-hand-side count
        _case(name="hypradon_batch12", call="batch", phase="hypradon", count=12, L_min=7, L_max=9, nrhs_max=16, draw=4),
        # scattered sources and targets
        _case(name="genradon2d_n512_points", call="points", L=9, nsrc=200003, ntgt=150001),
        # least squares with the operator and its adjoint
        _case(name="genradon2d_n512_cgls", call="cgls", L=9, iters=5),
    ]


# ----------------------------------------------------------------- work

def _batch_problems(case) -> list[tuple[int, int]]:
    """(L, right-hand sides) of the problems of a batch: sizes in turn, counts drawn."""
    rng = np.random.default_rng(case["draw"])
    span = case["L_max"] - case["L_min"] + 1
    return [(case["L_min"] + i % span, int(k)) for i, k in
            enumerate(rng.integers(1, case["nrhs_max"] + 1, size=case["count"]))]


def _apply_flops(d, L, q, phase, nrhs, tables=False) -> float:
    """Operations of one apply: every phase factor once (the reduced phase and its sine and
    cosine, the sine and cosine alone where the phases are kept), and per right-hand side the
    modulations, the factorised interpolation and the switch."""
    n, r = float(2 ** (L * d)), q ** d
    split = phase in ("dot", "separable")
    factors = n * (L * (2 ** d + 1) * r + (d * q * q if split else r * r))
    per = n * (L * ((2 ** (d + 1) - 2) * q ** (d + 1) * 4 + (2 ** d + 1) * r * 6)
               + 8 * (d * q ** (d + 1) if split else r * r))
    return factors * (18 if tables else 40) + nrhs * per


def _applies(case) -> int:
    return {"gradient": 2, "cgls": 2 * case.get("iters", 0) + 1}.get(case["call"], 1)


def work(case) -> dict:
    d, q, phase = case["d"], case["q"], case["phase"]
    c = 16 if case["precision"] == "fp64" else 8
    if case["call"] == "batch":
        probs = _batch_problems(case)
        return {"bytes": float(sum(2 * k * 2 ** (L * d) * c for L, k in probs)),
                "flops": sum(_apply_flops(d, L, q, phase, k) for L, k in probs)}
    n = 2 ** (case["L"] * d)
    pts = case["nsrc"] + case["ntgt"] if case["call"] == "points" else 2 * n
    return {"bytes": float(_applies(case) * case["nrhs"] * pts * c),
            "flops": _applies(case) * _apply_flops(d, case["L"], q, phase, case["nrhs"], bool(case.get("tables")))}


def _cost(case) -> float:
    """Rough relative run time: FP64 operations are many times dearer, and one-sided paths
    (FP64, space, adjoint) evaluate the phases for every right-hand side."""
    w = work(case)["flops"]
    if case["precision"] == "fp64":
        return 40 * w * case["nrhs"] ** 0.7
    if case["call"] in ("gradient", "points") or case["d"] == 3:
        return w * case["nrhs"] ** 0.5
    return w


# ----------------------------------------------------------------- drawn cases

def draw(rng) -> dict:
    limit = max(_cost(c) for c in listed() if c["precision"] != "fp64")
    call = rng.choice(["apply", "apply", "apply", "apply", "gradient", "gradient", "points", "batch", "cgls"])
    d = 3 if call in ("apply", "gradient") and rng.random() < 0.25 else 2
    case = _case(call=call, d=d, q=5 if d == 2 else 4)
    if rng.random() < 0.3:
        case["q"] = rng.choice([3, 4, 6, 8]) if d == 2 else 3
    case["phase"] = rng.choice(["genradon", "genradon", "hypradon", "hypradon", "dot"] if d == 2 else ["genradon", "genradon", "dot"])
    case["nrhs"] = 1 if rng.random() < 0.4 else int(round(math.exp(rng.uniform(math.log(2), math.log(16)))))
    if call == "batch":
        lo = rng.randint(6, 8)
        case.update(count=rng.randint(3, 14), L_min=lo, L_max=rng.randint(lo, 9), nrhs_max=rng.randint(2, 16), draw=rng.randint(0, 999))
        case.pop("nrhs")
        case["nrhs"] = 1
        case.pop("L")
        case["precision"] = rng.choice(["mixed", "mixed", "bf16x3"]) if case["q"] <= 5 else "mixed"
        while _cost(case) > limit:
            case["count"] -= 1
        return case
    case["L"] = rng.randint(5, 10) if d == 2 else rng.randint(3, 6)
    if call == "apply":
        pick = ["mixed", "mixed", "mixed", "fp64", "mixed_sfu"]
        if d == 2 and case["q"] <= 5 and case["nrhs"] > 1:
            pick += ["bf16x3", "tf32x3"]
        case["precision"] = rng.choice(pick)
        if case["precision"] == "mixed" and case["nrhs"] == 1 and case["q"] <= 5 and rng.random() < 0.3:
            case["tables"] = True
    elif call == "gradient":
        case["precision"] = rng.choice(["mixed", "mixed", "fp64"])
    elif call == "cgls":
        case.update(nrhs=1, iters=rng.randint(2, 6))
    if rng.random() < 0.2:
        case["off"] = 0.5
    if rng.random() < 0.15:
        case["node_kind"] = 1
    while True:
        if call == "points":
            n = 2 ** (2 * case["L"])
            case["nsrc"], case["ntgt"] = (int(n * math.exp(rng.uniform(-1.5, 0.5))) | 1 for _ in range(2))
        if _cost(case) <= limit:
            return case
        if case["nrhs"] > 4:
            case["nrhs"] //= 2
        else:
            case["L"] -= 1


# ----------------------------------------------------------------- inputs and plans

def _spec(case, L=None) -> workloads.Spec:
    L = case["L"] if L is None else L
    hyp = case["phase"] == "hypradon"
    kw = dict(scale=float(2 ** L), x_lo=(1.0, 0.0, 0.0), y_lo=(1.0, 0.0, 0.0), y_w=(1.0, 1.0, 1.0)) if hyp else {}
    off = case.get("off", 0.0)
    return workloads.Spec("case", case["d"], L, case["q"], case["phase"], precision=case["precision"],
                          node_kind=case.get("node_kind", 0), tgt_off=off, src_off=off, **kw)


def _dtype(case):
    return torch.complex128 if case["precision"] == "fp64" else torch.complex64


def _normal(gen, shape, dtype):
    """Real and imaginary parts N(0, 1), drawn in 64 bits and rounded."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64)).to(dtype)


def _points(spec, case, gen):
    """Half of the points spread evenly, half in clusters (8 per domain), inside the domains."""
    x_lo, x_w, y_lo, y_w = spec.domain()
    sets = []
    for n, lo, w in ((case["nsrc"], y_lo, y_w), (case["ntgt"], x_lo, x_w)):
        u = torch.rand(n, spec.d, generator=gen, device="cuda", dtype=torch.float64)
        mid = torch.rand(8, spec.d, generator=gen, device="cuda", dtype=torch.float64)
        pick = torch.randint(0, 8, (n,), generator=gen, device="cuda")
        near = (mid[pick] + 0.02 * torch.randn(n, spec.d, generator=gen, device="cuda", dtype=torch.float64)) % 1.0
        u = torch.where((torch.arange(n, device="cuda") % 2 == 0)[:, None], u, near).clamp(0.0, 1.0 - 1e-9)
        lo, w = (torch.tensor(v[: spec.d], dtype=torch.float64, device="cuda") for v in (lo, w))
        sets.append(lo + w * u)
    return sets


def _inputs(case, seed) -> dict:
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dt = _dtype(case)
    if case["call"] == "batch":
        return {"gs": [_normal(gen, (k, 2 ** (L * case["d"])), dt) for L, k in _batch_problems(case)]}
    spec = _spec(case)
    n, r = spec.npts, case["nrhs"]
    if case["call"] == "points":
        src, tgt = _points(spec, case, gen)
        return {"src": src, "tgt": tgt, "g": _normal(gen, (r, case["nsrc"]), dt)}
    if case["call"] == "cgls":
        # data of a sparse model: spikes at about one point in a hundred, and a little noise
        m = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
        m = m * (torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) < 0.01)
        return {"m": m.to(dt), "noise": _normal(gen, (n,), dt)}
    return {"g": _normal(gen, (r, n), dt), **({"u": _normal(gen, (r, n), dt)} if case["call"] == "gradient" else {})}


def prepare(case, seed):
    x = _inputs(case, seed)
    state = {"call": case["call"]}
    if case["call"] == "batch":
        probs = _batch_problems(case)
        state["plans"] = [bf.Plan.from_spec(_spec(case, L), max_nrhs=k) for L, k in probs]
        state.update(gs=x["gs"], fs=[torch.empty_like(g) for g in x["gs"]], nrhs=[k for _, k in probs])
        return state
    spec = _spec(case)
    if case["call"] == "points":
        state["plan"] = bf.Plan.from_spec(spec, max_nrhs=case["nrhs"], sources=x["src"].cpu().numpy(), targets=x["tgt"].cpu().numpy())
        state["g"] = x["g"]
        return state
    state["plan"] = bf.Plan.from_spec(spec, max_nrhs=case["nrhs"], phase_tables=bool(case.get("tables")))
    if case["call"] == "cgls":
        state.update(data=_cgls_data(case, x), iters=case["iters"])
    elif case["call"] == "gradient":
        state.update(g=x["g"].requires_grad_(), u=x["u"])
    else:
        state["g"] = x["g"]
    return state


def run(state):
    call = state["call"]
    if call == "batch":
        bf.apply_batched(state["plans"], state["gs"], state["fs"], state["nrhs"])
        return state["fs"]
    plan = state["plan"]
    if call == "gradient":
        f = autograd.butterfly(state["g"], plan)
        grad, = torch.autograd.grad(f, state["g"], state["u"])
        return {"f": f.detach(), "grad": grad}
    if call == "cgls":
        m, hist = autograd.cgls(plan, state["data"], iters=state["iters"])
        return {"m": m, "residuals": hist}
    return plan.apply(state["g"])


# ----------------------------------------------------------------- the same operator in 64 bits

def _sum_phase(kind, d, s, X, Y):
    """Phi in cycles from d target and d source coordinate tensors that broadcast."""
    two_pi = 2 * math.pi
    if kind == "dot":
        return s * sum(x * y for x, y in zip(X, Y))
    if kind == "hypradon":
        return s * X[0] * torch.sqrt(Y[0] ** 2 + (Y[1] * X[1]) ** 2)
    if d == 2:
        a = [(2 + torch.sin(two_pi * X[0]) * torch.sin(two_pi * X[1])) / 3,
             (2 + torch.cos(two_pi * X[0]) * torch.cos(two_pi * X[1])) / 3]
    else:
        a = [(2 + torch.sin(two_pi * X[k]) * torch.cos(two_pi * X[(k + 1) % 3])) / 3 for k in range(3)]
    return s * (sum(x * y for x, y in zip(X, Y)) + torch.sqrt(sum((ak * y) ** 2 for ak, y in zip(a, Y))))


class _Exact:
    """The butterfly in complex128.  Weights of level l: [rhs, a_0.., b_0.., t_0..] with 2^l target
    boxes, 2^(L-l) source boxes and q nodes per dimension."""

    def __init__(self, case, L=None):
        spec = _spec(case, L)
        self.d, self.L, self.q, self.kind, self.s = spec.d, spec.L, spec.q, spec.phase, spec.scale
        self.off, self.m = spec.tgt_off, spec.L // 2
        self.x_lo, self.x_w, self.y_lo, self.y_w = spec.domain()
        q = self.q
        j = torch.arange(q, dtype=torch.float64)
        z = 0.5 * torch.cos(j * math.pi / (q - 1)) if spec.node_kind == 0 else 0.5 * torch.cos((2 * j + 1) * math.pi / (2 * q))
        self.M = [self._lagrange(z, (z + h - 0.5) / 2).cuda().to(torch.complex128) for h in (0, 1)]   # [t][t']
        self.grid = self._lagrange(z, torch.tensor([self.off - 0.5], dtype=torch.float64))[:, 0].cuda()
        self.zh, self.z = z, z.cuda()

    @staticmethod
    def _lagrange(z, xi):
        rows = []
        for t in range(len(z)):
            v = torch.ones_like(xi)
            for k in range(len(z)):
                if k != t:
                    v = v * (xi - z[k]) / (z[t] - z[k])
            rows.append(v)
        return torch.stack(rows)

    # coordinates per dimension: box centres [n], nodes [n, q], grid points [n]
    def _boxes(self, lo, w, n):
        return lo + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * (w / n)

    def x(self, k, l):
        return self._boxes(self.x_lo[k], self.x_w[k], 2 ** l)

    def y(self, k, l):
        return self._boxes(self.y_lo[k], self.y_w[k], 2 ** (self.L - l))

    def xn(self, k, l):
        return self.x(k, l)[:, None] + self.x_w[k] / 2 ** l * self.z

    def yn(self, k, l):
        return self.y(k, l)[:, None] + self.y_w[k] / 2 ** (self.L - l) * self.z

    def shaped(self, v, k, box, nodes):
        """A [n] or [n, q] tensor of dimension k along axis `box` + k (0 targets, d sources), nodes along 2 d + k."""
        shape = [1] * (3 * self.d)
        shape[box + k] = v.shape[0]
        if nodes:
            shape[2 * self.d + k] = v.shape[1]
        return v.reshape(shape)

    def E(self, X, Y):
        th = _sum_phase(self.kind, self.d, self.s, X, Y)
        th = 2 * math.pi * (th - torch.round(th))
        return torch.complex(torch.cos(th), torch.sin(th))

    def contract(self, u, M, k, transpose):
        """sum over node axis k: M[t][t'] u(t') or, transposed, M[t][t'] u(t)."""
        ax = 1 + 2 * self.d + k
        return (u.movedim(ax, -1) @ (M if transpose else M.t())).movedim(-1, ax)

    def half(self, axis0, bits):
        """Index of every second box (`bits` per dimension) along the axes from axis0."""
        idx = [slice(None)] * (1 + 3 * self.d)
        for k, b in enumerate(bits):
            idx[axis0 + k] = slice(b, None, 2)
        return tuple(idx)

    def bits(self):
        return list(itertools.product((0, 1), repeat=self.d))

    def zeros(self, R, l):
        return torch.zeros([R] + [2 ** l] * self.d + [2 ** (self.L - l)] * self.d + [self.q] * self.d, dtype=torch.complex128, device="cuda")

    def level(self, w, l, adj):
        """Level l -> l + 1, or its conjugate transpose."""
        d, col = self.d, l < self.m
        out = self.zeros(w.shape[0], l if adj else l + 1)
        pre = {}
        for c in self.bits():
            src = self.half(1 + d, c)
            Yc = [self.shaped(self.yn(k, l)[c[k]::2] if col else self.y(k, l)[c[k]::2], k, d, col) for k in range(d)]
            if not col:
                pre = self.E([self.shaped(self.xn(k, l), k, 0, True) for k in range(d)], Yc)
                u0 = None if adj else pre.conj() * w[src]
                back = 0
            for a in self.bits():
                tgt = self.half(1, a)
                if col:
                    Xa = [self.shaped(self.x(k, l + 1)[a[k]::2], k, 0, False) for k in range(d)]
                    e_in = self.E(Xa, Yc)
                    e_out = self.E(Xa, [self.shaped(self.yn(k, l + 1), k, d, True) for k in range(d)])
                    v = e_out * w[tgt] if adj else e_in * w[src]
                    for k in range(d):
                        v = self.contract(v, self.M[c[k]], k, adj)
                    if adj:
                        out[src] += e_in.conj() * v
                    else:
                        out[tgt] += e_out.conj() * v
                else:
                    e_out = self.E([self.shaped(self.xn(k, l + 1)[a[k]::2], k, 0, True) for k in range(d)], Yc)
                    v = e_out.conj() * w[tgt] if adj else u0
                    for k in range(d):
                        v = self.contract(v, self.M[a[k]], k, not adj)
                    if adj:
                        back = back + v
                    else:
                        out[tgt] += e_out * v
            if not col and adj:
                out[src] = pre * back
        return out

    def switch(self, w, adj):
        d, l = self.d, self.m
        out = torch.zeros_like(w)
        Y = [self.shaped(self.yn(k, l), k, d, True) for k in range(d)]
        nodes = tuple(range(1 + 2 * d, 1 + 3 * d))
        for s in itertools.product(range(self.q), repeat=d):
            e = self.E([self.shaped(self.xn(k, l)[:, s[k]], k, 0, False) for k in range(d)], Y)
            at = (Ellipsis, *s)
            if adj:
                out += e.conj() * w[at].reshape(list(w.shape[:1 + 2 * d]) + [1] * d)
            else:
                out[at] = (e * w).sum(dim=nodes)
        return out

    def ends(self, first):
        """Factors [boxes, nodes] and [boxes] of the first step (sources) or the last (targets)."""
        d, lag = self.d, 1.0
        for k in range(d):
            lag = lag * self.shaped(self.grid[None], k, 0, True)
        if first:
            X = [self.shaped(self.x(k, 0), k, 0, False) for k in range(d)]
            pt = [self.shaped(self.y_lo[k] + (torch.arange(2 ** self.L, dtype=torch.float64, device="cuda") + self.off) * (self.y_w[k] / 2 ** self.L), k, d, False) for k in range(d)]
            return lag * self.E(X, [self.shaped(self.yn(k, 0), k, d, True) for k in range(d)]).conj(), self.E(X, pt)
        Y = [self.shaped(self.y(k, self.L), k, d, False) for k in range(d)]
        pt = [self.shaped(self.x_lo[k] + (torch.arange(2 ** self.L, dtype=torch.float64, device="cuda") + self.off) * (self.x_w[k] / 2 ** self.L), k, 0, False) for k in range(d)]
        return lag * self.E([self.shaped(self.xn(k, self.L), k, 0, True) for k in range(d)], Y).conj(), self.E(pt, Y)

    def sweep(self, w, adj):
        for l in range(self.L) if not adj else reversed(range(self.L)):
            if l == self.m and not adj:
                w = self.switch(w, False)
            w = self.level(w, l, adj)
            if l == self.m and adj:
                w = self.switch(w, True)
        return w

    def apply(self, g):
        R, d, N = g.shape[0], self.d, 2 ** self.L
        node, pt = self.ends(True)
        w = node * (pt * g.to(torch.complex128).reshape([R] + [1] * d + [N] * d + [1] * d))
        w = self.sweep(w, False)
        node, pt = self.ends(False)
        w = (node * w).sum(dim=tuple(range(1 + 2 * d, 1 + 3 * d)), keepdim=True)
        return (pt * w).reshape(R, -1)

    def adjoint(self, f):
        R, d, N = f.shape[0], self.d, 2 ** self.L
        node, pt = self.ends(False)
        w = node.conj() * (pt.conj() * f.to(torch.complex128).reshape([R] + [N] * d + [1] * 2 * d))
        w = self.sweep(w, True)
        node, pt = self.ends(True)
        w = (node.conj() * w).sum(dim=tuple(range(1 + 2 * d, 1 + 3 * d)), keepdim=True)
        return (pt.conj() * w).reshape(R, -1)

    def _leaf(self, pts, lo, w):
        """Leaf box index per dimension and Lagrange values [n, q] per dimension of points [n, d]."""
        N, idx, lag = 2 ** self.L, [], []
        for k in range(self.d):
            h = w[k] / N
            i = torch.floor((pts[:, k] - lo[k]) / h).clamp(0, N - 1)
            xi = (pts[:, k] - (lo[k] + (i + 0.5) * h)) / h
            idx.append(i.long())
            lag.append(self._lagrange(self.zh, xi).t())
        flat = idx[0]
        for i in idx[1:]:
            flat = flat * N + i
        nodes = lag[0]
        for v in lag[1:]:
            nodes = nodes[..., None] * v.reshape([len(v)] + [1] * (nodes.dim() - 1) + [self.q])
        return flat, nodes

    def apply_points(self, g, src, tgt):
        R, d, N, q = g.shape[0], self.d, 2 ** self.L, self.q
        xc = [torch.tensor(self.x_lo[k] + 0.5 * self.x_w[k], dtype=torch.float64, device="cuda") for k in range(d)]
        yc = [torch.tensor(self.y_lo[k] + 0.5 * self.y_w[k], dtype=torch.float64, device="cuda") for k in range(d)]
        box, lag = self._leaf(src, self.y_lo, self.y_w)
        v = self.E(xc, [src[:, k] for k in range(d)]) * g.to(torch.complex128)
        w = torch.zeros(R, N ** d, q ** d, dtype=torch.complex128, device="cuda")
        w.index_add_(1, box, v[:, :, None] * lag.reshape(1, len(box), -1))
        w = w.reshape([R] + [1] * d + [N] * d + [q] * d)
        w = w * self.E([self.shaped(self.x(k, 0), k, 0, False) for k in range(d)], [self.shaped(self.yn(k, 0), k, d, True) for k in range(d)]).conj()
        w = self.sweep(w, False)
        w = w * self.E([self.shaped(self.xn(k, self.L), k, 0, True) for k in range(d)], [self.shaped(self.y(k, self.L), k, d, False) for k in range(d)]).conj()
        box, lag = self._leaf(tgt, self.x_lo, self.x_w)
        w = (w.reshape(R, N ** d, q ** d)[:, box] * lag.reshape(1, len(box), -1)).sum(dim=2)
        return self.E([tgt[:, k] for k in range(d)], yc) * w


def _cgls_data(case, x):
    """Data that the least-squares solve is given: a smooth random mix of the spikes and noise."""
    n = 2 ** case["L"]
    m = torch.fft.fft2(x["m"].reshape(n, n)).reshape(-1)
    return (m + 0.05 * torch.linalg.vector_norm(m) / n * x["noise"]).to(_dtype(case))


def _cgls(op, data, iters):
    m = torch.zeros_like(data)
    r = data.clone()
    s = op.adjoint(r[None])[0]
    p, gamma = s.clone(), torch.vdot(s, s).real
    hist = [torch.linalg.vector_norm(r).item()]
    for _ in range(iters):
        t = op.apply(p[None])[0]
        alpha = gamma / torch.vdot(t, t).real
        m = m + alpha * p
        r = r - alpha * t
        s = op.adjoint(r[None])[0]
        new = torch.vdot(s, s).real
        p, gamma = s + (new / gamma) * p, new
        hist.append(torch.linalg.vector_norm(r).item())
    return m, hist


def exact(case, seed):
    x = _inputs(case, seed)
    if case["call"] == "batch":
        return [_Exact(case, L).apply(g) for (L, _), g in zip(_batch_problems(case), x["gs"])]
    op = _Exact(case)
    if case["call"] == "points":
        return op.apply_points(x["g"], x["src"], x["tgt"])
    if case["call"] == "cgls":
        m, hist = _cgls(op, _cgls_data(case, x).to(torch.complex128), case["iters"])
        return {"m": m, "residuals": hist}
    if case["call"] == "gradient":
        return {"f": op.apply(x["g"]), "grad": op.adjoint(x["u"])}
    return op.apply(x["g"])
