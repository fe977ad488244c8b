"""The work that users of this package have it do, as measurable cases.

Every case goes through the public binding (``paper_0810_0330_gb300.binding``)
or the autograd entry (``adjoint.wilson_seed_solve``).  Sizes, tolerances and
parameters are those of the benchmark, the workload configurations and the
tests of this repository.  Mixed-precision solves run to 1e-12 (the tolerance
of the mixed-precision gradient tests), FP64 solves to the benchmark's 1e-8
(1e-12 for the seed system).

``listed()`` are the fixed cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes inputs and contexts, ``run`` is one pass, ``work`` its
algorithmic bytes and operations, ``exact`` its result from plain torch in
64 bits.
"""
import math

import torch

from paper_0810_0330_gb300 import binding as S
from paper_0810_0330_gb300.adjoint import wilson_seed_solve

DEV = "cuda"


def listed():
    return [
        # One operator application to one vector of a small lattice: the latency
        # of a single call inside a caller's own Krylov loop.
        _wapply("apply_wilson_4x4x4x4", (4, 4, 4, 4), op=0, bc_t=1, cols=1),
        # The normal operator on a block of spinors of a production-sized lattice
        # (residual checks, callers' own block solvers).
        _wapply("apply_wilson_16x16x16x16_12cols", (16, 16, 16, 16), op=0, bc_t=0, cols=12),
        # The FP32 copy of the operator on the caller's own layout.
        _wapply("apply_wilson_fp32_16x16x16x32_12cols", (16, 16, 16, 32), op=3, bc_t=0, cols=12),
        # CSR matrix times vector beyond the L2 cache.
        _capply("apply_csr_laplacian_2048sq", (2048, 2048), shift=0.0, cols=1),
        # The benchmark: a propagator (12 point sources) on 8^4 in FP64.
        _wsolve("solve_wilson_8x8x8x8_fp64", (8, 8, 8, 8), "point", precision=0),
        # The same propagator in mixed precision.
        _wsolve("solve_wilson_8x8x8x8_mixed", (8, 8, 8, 8), "point", precision=1),
        # Noise sources on the large lattice, mixed precision.
        _wsolve("solve_wilson_16x16x16x32_mixed", (16, 16, 16, 32), "z4", precision=1, m_max=1000),
        # A small real problem with full reorthogonalization.
        _csolve("solve_laplacian_64x64_full_reorth", (64, 64), shift=0.0, nrhs=4, m_max=1000, freq=1, tol_seed=1e-12),
        # An ordinary real problem: shifted 3-d Laplacian, several right-hand sides.
        _csolve("solve_csr_48x48x48_fp64", (48, 48, 48), shift=0.05, nrhs=8, m_max=500, freq=100, tol_seed=1e-10),
        # Training step through the solve: loss, gradients for b and kappa, 16^4.
        _adjoint("adjoint_wilson_16x16x16x16_fp64", (16, 16, 16, 16), nrhs=8, precision=0),
        # Many uneven problems at once.
        _batch("batch_csr_12_problems_fp64", count=12, n_min=1e4, n_max=2.5e5, precision=0),
    ]


def draw(rng):
    kind = rng.choice(["wapply", "wapply", "capply", "wsolve", "wsolve", "wsolve", "csolve", "reorth", "adjoint", "batch"])
    if kind == "wapply":
        op = rng.choice([0, 0, 1, 2, 3, 4, 5])
        c = _wapply("", _lattice(rng, 256, 131072), op=op, bc_t=rng.randint(0, 1), cols=_logint(rng, 1, 12))
        c["kappa"] = round(rng.uniform(0.12, 0.16), 4)
    elif kind == "capply":
        c = _capply("", (_logint(rng, 48, 2048), _logint(rng, 48, 2048)), shift=round(rng.uniform(0.0, 1.0), 3),
                    cols=_logint(rng, 1, 8))
    elif kind == "wsolve":
        precision = rng.randint(0, 1)
        c = _wsolve("", _lattice(rng, 256, 65536 if precision else 8192), rng.choice(["point", "z4", "gauss"]),
                    precision=precision, nrhs=rng.randint(2, 12), m_max=1000, freq=rng.choice([25, 50, 100]))
        c["bc_t"] = rng.randint(0, 1)
    elif kind == "csolve":
        d = rng.choice([2, 3])
        n = _loguniform(rng, 1e4, 2.5e5)
        sides = tuple(max(8, int(round(n ** (1.0 / d) * rng.uniform(0.8, 1.2)))) for _ in range(d))
        c = _csolve("", sides, shift=round(rng.uniform(0.03, 1.0), 3), nrhs=rng.randint(2, 16), m_max=500,
                    freq=rng.choice([25, 100]), tol_seed=1e-10)
    elif kind == "reorth":
        c = _csolve("", (_logint(rng, 24, 72), _logint(rng, 24, 72)), shift=round(rng.uniform(0.0, 0.05), 3),
                    nrhs=rng.randint(2, 8), m_max=1000, freq=rng.choice([1, 1, 2, 5]), tol_seed=1e-12)
    elif kind == "adjoint":
        c = _adjoint("", _lattice(rng, 256, 32768), nrhs=rng.randint(1, 8), precision=rng.randint(0, 1))
        c["bc_t"] = rng.randint(0, 1)
    else:
        c = _batch("", count=rng.randint(3, 12), n_min=1e4, n_max=1.5e5, precision=0)
        c["variant"] = rng.randint(1, 1 << 20)
    del c["name"]
    return c


# --- case descriptions -------------------------------------------------------

def _wilson(name, kind, dims, kappa, bc_t):
    return {"name": name, "kind": kind, "X": dims[0], "Y": dims[1], "Z": dims[2], "T": dims[3], "kappa": kappa, "bc_t": bc_t}


def _wapply(name, dims, op, bc_t, cols):
    return dict(_wilson(name, "wilson_apply", dims, 0.155, bc_t), op=op, cols=cols)


def _wsolve(name, dims, sources, precision, nrhs=12, m_max=3000, freq=100):
    return dict(_wilson(name, "wilson_solve", dims, 0.155, 0), sources=sources, precision=precision, nrhs=nrhs,
                m_max=m_max, freq=freq, tol_seed=1e-12, tol_rest=1e-12 if precision else 1e-8)


def _adjoint(name, dims, nrhs, precision):
    return dict(_wilson(name, "adjoint", dims, 0.150, 0), nrhs=nrhs, precision=precision, m_max=1000, freq=100,
                tol_seed=1e-12 if precision else 1e-10, tol_rest=1e-12 if precision else 1e-8)


def _grid(name, kind, sides, shift):
    s = tuple(sides) + (1,) * (3 - len(sides))
    return {"name": name, "kind": kind, "n1": s[0], "n2": s[1], "n3": s[2], "d": len(sides), "shift": shift}


def _capply(name, sides, shift, cols):
    return dict(_grid(name, "csr_apply", sides, shift), cols=cols)


def _csolve(name, sides, shift, nrhs, m_max, freq, tol_seed):
    return dict(_grid(name, "csr_solve", sides, shift), nrhs=nrhs, m_max=m_max, freq=freq, precision=0,
                tol_seed=tol_seed, tol_rest=1e-8)


def _batch(name, count, n_min, n_max, precision):
    return {"name": name, "kind": "batch", "count": count, "n_min": n_min, "n_max": n_max, "precision": precision,
            "variant": 0, "m_max": 500, "freq": 100, "tol_seed": 1e-10, "tol_rest": 1e-8}


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(_loguniform(rng, lo, hi)))))


def _lattice(rng, lo, hi):
    """Four dimensions, odd ones among them, with a volume spread over lo..hi."""
    vol = _loguniform(rng, lo, hi)
    side = vol ** 0.25
    x, y, z = (max(2, int(round(side * rng.uniform(0.7, 1.4)))) for _ in range(3))
    t = max(2, int(vol / (x * y * z)))
    while x * y * z * t > hi and x > 2:
        x -= 1
    return x, y, z, t


def _batch_grids(case):
    """(sides, shift, nrhs) of each problem: 2-d or 3-d, n log-uniform, 4..16 right-hand sides."""
    import random
    rng = random.Random(case["variant"])
    out = []
    for _ in range(case["count"]):
        n = _loguniform(rng, case["n_min"], case["n_max"])
        d = rng.choice([2, 3])
        side = max(2, int(round(n ** (1.0 / d))))
        out.append(((side,) * d, rng.uniform(0.01, 1.0), rng.randint(4, 16)))
    return out


# --- inputs --------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape, cplx=False):
    if cplx:
        return torch.complex(torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64),
                             torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64))
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _dims(case):
    return case["X"], case["Y"], case["Z"], case["T"]


def _sites(case):
    return case["X"] * case["Y"] * case["Z"] * case["T"]


def _links(case, g):
    """exp(0.3 i H), H random Hermitian traceless: [mu][site][3][3]."""
    m = _randn(g, 4 * _sites(case), 3, 3, cplx=True)
    h = 0.5 * (m + m.mH)
    h = h - (torch.einsum("kaa->k", h).real / 3.0)[:, None, None] * torch.eye(3, device=DEV, dtype=h.dtype)
    # exp by Taylor series of a quarter of the exponent, squared twice
    a, e = 0.075j * h, torch.eye(3, device=DEV, dtype=h.dtype).expand_as(h)
    term = e
    for k in range(1, 19):
        term = _mul3(term, a) / k
        e = e + term
    e = _mul3(e, e)
    U = _mul3(e, e).reshape(4, _sites(case), 3, 3).contiguous()
    torch.cuda.synchronize()   # a context reads its links while it is created, on a stream of its own
    return U


def _mul3(a, b):
    """Products of stacks a [k][.][3] and b [k][3][.], element by element (batched
    library products are limited in the size of a stack)."""
    return sum(a[:, :, c, None] * b[:, c, None, :] for c in range(3))


def _sources(case, g):
    """Right-hand side block, as its (ncols, n) transpose."""
    n, p = 12 * _sites(case), case["nrhs"]
    if case["sources"] == "point":
        site = int(torch.randint(0, _sites(case), (1,), generator=g, device=DEV))
        e = torch.zeros(p, n, dtype=torch.complex128, device=DEV)
        for j in range(p):
            e[j, 12 * site + j % 12] = 1.0
        return e
    if case["sources"] == "z4":
        k = torch.randint(0, 4, (p, n), generator=g, device=DEV)
        return torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device=DEV)[k]
    return _randn(g, p, n, cplx=True)


def _params(case, **kw):
    return S.seed_params_default(m_max=case["m_max"], reorth_freq=case["freq"], reorth_passes=2, x0_zero=1,
                                 tol_seed=case["tol_seed"], tol_rest=case["tol_rest"], precision=case["precision"], **kw)


def _grid_csr(sides, shift):
    """Dirichlet Laplacian (2d on the diagonal, -1 per neighbour) plus shift, as CSR arrays on the GPU."""
    n = math.prod(sides)
    idx = torch.arange(n, device=DEV)
    cols, ok, vals, stride = [idx], [torch.ones(n, dtype=torch.bool, device=DEV)], [2.0 * len(sides) + shift], 1
    for s in sides:
        i = (idx // stride) % s
        cols = [idx - stride] + cols + [idx + stride]
        ok = [i > 0] + ok + [i < s - 1]
        vals = [-1.0] + vals + [-1.0]
        stride *= s
    ok = torch.stack(ok, 1)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(ok.sum(1), 0, out=rp[1:])
    ci = torch.stack(cols, 1)[ok]
    v = torch.tensor(vals, dtype=torch.float64, device=DEV).expand(n, -1)[ok]
    return rp.int(), ci.int(), v.contiguous()


def _sides(case):
    return (case["n1"], case["n2"], case["n3"])[:case["d"]]


# --- one pass --------------------------------------------------------------------

def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "wilson_apply":
        low = case["op"] >= 3
        ctx = S.seed_create_wilson(_dims(case), case["kappa"], _links(case, g),
                                   S.seed_params_default(m_max=4, precision=1 if low else 0), bc_t=case["bc_t"])
        x = _randn(g, case["cols"], 12 * _sites(case), cplx=True)
        x = x.to(torch.complex64) if low else x
        return {"case": case, "ctx": ctx, "X": x.t(), "Y": torch.empty_like(x).t()}
    if kind == "csr_apply":
        rp, ci, v = _grid_csr(_sides(case), case["shift"])
        ctx = S.seed_create_csr(rp, ci, v, S.seed_params_default(m_max=4))
        x = _randn(g, case["cols"], rp.shape[0] - 1)
        return {"case": case, "ctx": ctx, "X": x.t(), "Y": torch.empty_like(x).t()}
    if kind == "wilson_solve":
        ctx = S.seed_create_wilson(_dims(case), case["kappa"], _links(case, g), _params(case), bc_t=case["bc_t"])
        eta = _sources(case, g)
        return {"case": case, "ctx": ctx, "eta": eta.t(), "B": torch.empty_like(eta).t(), "X": torch.empty_like(eta).t()}
    if kind == "csr_solve":
        rp, ci, v = _grid_csr(_sides(case), case["shift"])
        b = _randn(g, case["nrhs"], rp.shape[0] - 1)
        return {"case": case, "ctx": S.seed_create_csr(rp, ci, v, _params(case)), "B": b.t(), "X": torch.empty_like(b).t()}
    if kind == "adjoint":
        U, n = _links(case, g), 12 * _sites(case)
        return {"case": case, "U": U, "B": _randn(g, case["nrhs"], n, cplx=True).t(),
                "T": _randn(g, case["nrhs"], n, cplx=True).t()}
    ctxs, Bs, Xs = [], [], []
    for sides, shift, nrhs in _batch_grids(case):
        rp, ci, v = _grid_csr(sides, shift)
        b = _randn(g, nrhs, rp.shape[0] - 1)
        ctxs.append(S.seed_create_csr(rp, ci, v, _params(case)))
        Bs.append(b.t())
        Xs.append(torch.empty_like(b).t())
    return {"case": case, "ctxs": ctxs, "B": Bs, "X": Xs}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("wilson_apply", "csr_apply"):
        S.seed_apply(state["ctx"], case.get("op", 0), state["X"], state["Y"])
        return state["Y"]
    if kind == "wilson_solve":
        # b = D^H eta turns D x = eta into the normal equations
        S.seed_apply(state["ctx"], 2, state["eta"], state["B"])
    if kind in ("wilson_solve", "csr_solve"):
        S.seed_solve_first(state["ctx"], state["B"], state["X"])
        S.seed_solve_rest(state["ctx"], state["B"], state["X"])
        return state["X"]
    if kind == "adjoint":
        kappa = torch.tensor(case["kappa"], dtype=torch.float64, requires_grad=True)
        B = state["B"].detach().requires_grad_(True)
        prm = dict(m_max=case["m_max"], reorth_freq=case["freq"], reorth_passes=2, tol_seed=case["tol_seed"],
                   tol_rest=case["tol_rest"], precision=case["precision"])
        X = wilson_seed_solve(kappa, B, state["U"], _dims(case), case["bc_t"], prm)
        loss = ((X - state["T"]).abs() ** 2).sum()
        loss.backward()
        return {"X": X.detach(), "dB": B.grad, "dkappa": kappa.grad}
    S.seed_batch_solve(state["ctxs"], state["B"], state["X"])
    return state["X"]


# --- algorithmic work ------------------------------------------------------------

def work(case):
    """Bytes: operator, inputs and outputs once.  Operations of a solve: the
    operator applications of its iterations (about 20 per decade of the residual
    on these Wilson operators, sqrt(condition)/2 * ln(2/tol) on the Laplacians)
    plus 10 per real element for the vector updates of an iteration."""
    kind = case["kind"]
    if kind == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for sides, shift, nrhs in _batch_grids(case):
            w = work(dict(_csolve("", sides, shift, nrhs, case["m_max"], case["freq"], case["tol_seed"])))
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    if kind.startswith("csr"):
        sides = _sides(case)
        n = math.prod(sides)
        nnz = n + 2 * sum(n // s * (s - 1) for s in sides)
        cols = case.get("cols") or case["nrhs"]
        b = 12.0 * nnz + 4.0 * (n + 1) + 16.0 * n * cols
        if kind == "csr_apply":
            return {"bytes": b, "flops": 2.0 * nnz * cols}
        low = sum(2.0 - 2.0 * math.cos(math.pi / (s + 1)) for s in sides) + case["shift"]
        its = 0.5 * math.sqrt((4.0 * len(sides) + case["shift"]) / low) * math.log(2.0 / case["tol_rest"])
        return {"bytes": b, "flops": its * cols * (2.0 * nnz + 10.0 * n)}
    vol = _sites(case)
    low = kind == "wilson_apply" and case["op"] >= 3
    cols, esz = case.get("cols") or case["nrhs"], 8 if low else 16
    b = 36.0 * esz * vol + 24.0 * esz * vol * cols
    apply_flops = 2 * 1368.0 * vol
    if kind == "wilson_apply":
        return {"bytes": b, "flops": apply_flops * cols * (1.0 if case["op"] in (0, 3) else 0.5)}
    its = 20.0 * (cols - 1) * -math.log10(case["tol_rest"]) - 20.0 * math.log10(case["tol_seed"])
    flops = its * (apply_flops + 240.0 * vol)
    if kind == "adjoint":   # the backward solves and the target block
        flops += 20.0 * cols * -math.log10(case["tol_rest"]) * (apply_flops + 240.0 * vol)
        b += 24.0 * esz * vol * cols
    return {"bytes": b, "flops": flops}


# --- the same results from plain torch in 64 bits ----------------------------------

def _gammas():
    i = 1j
    blocks = [[[0, i], [i, 0]], [[0, -1], [1, 0]], [[i, 0], [0, -i]], [[1, 0], [0, 1]]]
    out = []
    for b in blocks:
        B = torch.tensor(b, dtype=torch.complex128, device=DEV)
        g = torch.zeros(4, 4, dtype=torch.complex128, device=DEV)
        g[:2, 2:] = B
        g[2:, :2] = B.mH
        out.append(g)
    return out


class _Dirac:
    """D = 1 - kappa H on blocks (ncols, n)."""

    def __init__(self, case, U):
        self.X, self.Y, self.Z, self.T = _dims(case)
        self.kappa, self.bc = case["kappa"], case["bc_t"]
        self.U = U.reshape(4, -1, 3, 3)
        self.nbr = []
        s = torch.arange(_sites(case), device=DEV).reshape(self.T, self.Z, self.Y, self.X)
        for mu in range(4):
            self.nbr.append((torch.roll(s, -1, 3 - mu).reshape(-1), torch.roll(s, 1, 3 - mu).reshape(-1)))
        t = s // (self.X * self.Y * self.Z)
        one = torch.ones_like(t, dtype=torch.float64)
        self.sf = torch.where((t == self.T - 1) & bool(self.bc), -one, one).reshape(-1, 1, 1)
        self.sb = torch.where((t == 0) & bool(self.bc), -one, one).reshape(-1, 1, 1)
        eye = torch.eye(4, dtype=torch.complex128, device=DEV)
        self.proj = [(eye - g, eye + g) for g in _gammas()]

    def hop(self, v, dagger=False):
        p = v.shape[0]
        psi = v.reshape(p, -1, 4, 3).permute(1, 3, 0, 2).reshape(-1, 3, p * 4)   # [site][colour][column, spin]
        out = torch.zeros_like(psi)
        for mu in range(4):
            f, b = self.nbr[mu]
            pf, pb = self.proj[mu] if not dagger else self.proj[mu][::-1]
            hf = _mul3(self.U[mu], psi[f])
            hb = _mul3(self.U[mu][b].mH, psi[b])
            if mu == 3:
                hf, hb = hf * self.sf, hb * self.sb
            out += (hf.reshape(-1, 4) @ pf.t()).reshape(psi.shape)
            out += (hb.reshape(-1, 4) @ pb.t()).reshape(psi.shape)
        return out.reshape(-1, 3, p, 4).permute(2, 0, 3, 1).reshape(p, -1)

    def D(self, v, dagger=False):
        return v - self.kappa * self.hop(v, dagger)

    def A(self, v):
        return self.D(self.D(v), True)


def _solve(A, B):
    """A x = b for every row of B to rounding: CG, then CG again on the true residual."""
    X = torch.zeros_like(B)
    bn = torch.linalg.vector_norm(B, dim=1, keepdim=True)
    for _ in range(2):
        R = B - A(X) if X.any() else B.clone()
        P, E = R.clone(), torch.zeros_like(B)
        rho = torch.linalg.vecdot(R, R).real[:, None]
        stop = 1e-11 * torch.sqrt(rho)
        for it in range(6000):
            Q = A(P)
            a = rho / torch.linalg.vecdot(P, Q).real[:, None].clamp_min(1e-300)
            E += a * P
            R -= a * Q
            new = torch.linalg.vecdot(R, R).real[:, None]
            P = R + (new / rho.clamp_min(1e-300)) * P
            rho = new
            if it % 16 == 15 and bool((torch.sqrt(rho) <= stop.clamp_min(1e-17 * bn.max())).all()):
                break
        X = X + E
    return X


def _csr_op(rp, ci, v):
    M = torch.sparse_csr_tensor(rp.long(), ci.long(), v, size=(rp.shape[0] - 1,) * 2)
    return lambda x: (M @ x.t().contiguous()).t()


def exact(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "csr_apply":
        rp, ci, v = _grid_csr(_sides(case), case["shift"])
        return _csr_op(rp, ci, v)(_randn(g, case["cols"], rp.shape[0] - 1)).t()
    if kind == "csr_solve":
        rp, ci, v = _grid_csr(_sides(case), case["shift"])
        return _solve(_csr_op(rp, ci, v), _randn(g, case["nrhs"], rp.shape[0] - 1)).t()
    if kind == "batch":
        out = []
        for sides, shift, nrhs in _batch_grids(case):
            rp, ci, v = _grid_csr(sides, shift)
            out.append(_solve(_csr_op(rp, ci, v), _randn(g, nrhs, rp.shape[0] - 1)).t())
        return out
    op = _Dirac(case, _links(case, g))
    if kind == "wilson_apply":
        x = _randn(g, case["cols"], 12 * _sites(case), cplx=True)
        if case["op"] >= 3:
            x = x.to(torch.complex64).to(torch.complex128)
        y = op.A(x) if case["op"] % 3 == 0 else op.D(x, dagger=case["op"] % 3 == 2)
        return y.t()
    if kind == "wilson_solve":
        if _sites(case) * case["nrhs"] > 600000:
            return None   # minutes in plain torch
        return _solve(op.A, op.D(_sources(case, g), True)).t()
    n = 12 * _sites(case)
    B, T = _randn(g, case["nrhs"], n, cplx=True), _randn(g, case["nrhs"], n, cplx=True)
    X = _solve(op.A, B)
    lam = _solve(op.A, 2.0 * (X - T))
    # dA/dkappa = -(H^H D + D^H H); dL/dkappa = -Re <lambda, (dA/dkappa) x>
    dk = torch.linalg.vecdot(op.hop(lam), op.D(X)).real.sum() + torch.linalg.vecdot(op.D(lam), op.hop(X)).real.sum()
    return {"X": X.t(), "dB": lam.t(), "dkappa": dk}
