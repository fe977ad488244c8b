"""The FP64 Wilson operator in fixed-point arithmetic (csrc/wilson_fixed.cuh)
against an extended-precision reference, and against the FP64 kernel that
seed_wilson_apply_noalloc still runs.

Tolerances, derived.  With S = max over the nine terms of a site (its own
block, and per hop |kappa| times the link's largest row or column sum of
|Re| + |Im| times the neighbour block's largest real), the common exponent has
2^E <= 8 S (a factor 2 each from the exponents of spinor, kappa and row sum).
Per hop, in units of 2^-58 2^E: 12 for the dropped low products, 16 for the
link's rounding, 4 for the spinor's cut-off, 1.5 for the two shifts; times 8
hops, plus 1: at most 269 units, 2^-46.9 S, plus the rounding of the result,
2^-53 of it (D; D^H D doubles the count through the intermediate block).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
CLD = np.clongdouble


def gammas():
    B = [np.array([[0, 1j], [1j, 0]]), np.array([[0, -1], [1, 0]]), np.array([[1j, 0], [0, -1j]]), np.eye(2)]
    out = []
    for b in B:
        g = np.zeros((4, 4), dtype=complex)
        g[:2, 2:] = b
        g[2:, :2] = b.conj().T
        out.append(g)
    return out


def dirac(dims, kappa, bc_t, U, psi, sign):
    """(D psi, S) in extended precision; S per site, the scale of the bound above."""
    X, Y, Z, T = dims
    vol = X * Y * Z * T
    s = np.arange(vol).reshape(T, Z, Y, X)
    p = psi.reshape(vol, 4, 3).astype(CLD)
    Ul = U.astype(CLD)
    out = np.zeros_like(p)
    mx = np.maximum(np.abs(p.real), np.abs(p.imag)).reshape(vol, 12).max(1)
    scale = mx.copy()
    t = s // (X * Y * Z)   # site's t coordinate
    ab = np.abs(U.real) + np.abs(U.imag)
    l1 = np.maximum(ab.sum(2).max(2), ab.sum(3).max(2))   # [mu][site]
    for mu, g in enumerate(gammas()):
        f, b = np.roll(s, -1, 3 - mu).ravel(), np.roll(s, 1, 3 - mu).ravel()
        sf = np.where((t == T - 1) & bool(bc_t) & (mu == 3), -1, 1).ravel()[:, None, None]
        sb = np.where((t == 0) & bool(bc_t) & (mu == 3), -1, 1).ravel()[:, None, None]
        pf, pb = (np.eye(4) - sign * g).astype(CLD), (np.eye(4) + sign * g).astype(CLD)
        hf = np.einsum("vab,vsb->vsa", Ul[mu], p[f]) * sf
        hb = np.einsum("vba,vsb->vsa", Ul[mu][b].conj(), p[b]) * sb
        out += np.einsum("st,vta->vsa", pf, hf) + np.einsum("st,vta->vsa", pb, hb)
        scale = np.maximum(scale, np.maximum(abs(kappa) * l1[mu] * mx[f], abs(kappa) * l1[mu][b] * mx[b]))
    return (p - LD(kappa) * out).reshape(-1), scale


def blocks(kind, rng, vol, cols):
    x = rng.standard_normal((cols, vol, 12)) + 1j * rng.standard_normal((cols, vol, 12))
    if kind == "site_scales":      # neighbours further apart than 64 bits
        x *= 2.0 ** rng.integers(-120, 120, (cols, vol, 1))
    elif kind == "component_scales":
        x *= 2.0 ** rng.integers(-70, 1, (cols, vol, 12))
    elif kind == "point":
        x *= 0
        x[:, rng.integers(vol), 5] = 1.0
    elif kind == "sparse":
        x *= rng.uniform(size=(cols, vol, 1)) < 0.2
    elif kind == "extreme":        # beyond the blocks' exponent range: the FP64 form
        x *= 2.0 ** rng.choice([-1000, -690, 0, 690, 1000], (cols, vol, 1))
    return x.reshape(cols, -1)


def links(kind, rng, dims):
    from paper_0810_0330_gb300 import inputs as I
    U = I.random_su3_links(dims, 0.3, seed=3)
    if kind == "general":
        U = rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape)
        U = U * 2.0 ** rng.integers(-20, 20, U.shape[:2] + (1, 1))
    elif kind == "some_zero":
        U = U * (rng.uniform(size=U.shape[:2] + (1, 1)) < 0.5)
    elif kind == "unit":
        U = I.unit_links(dims)
    elif kind == "extreme":
        U = U * 2.0 ** rng.choice([-200, 0, 200], U.shape[:2] + (1, 1))
    return np.ascontiguousarray(U)


def on_gpu(seedlib, dims, kappa, bc_t, U, x, op):
    import torch
    ctx = seedlib.seed_create_wilson(dims, kappa, torch.from_numpy(U).cuda(), seedlib.seed_params_default(m_max=2),
                                     bc_t=bc_t)
    X = torch.from_numpy(x).cuda().t()
    Y = torch.empty_like(X.t()).t()
    seedlib.seed_apply(ctx, op, X, Y)
    torch.cuda.synchronize()
    seedlib.seed_destroy(ctx)
    return Y.t().cpu().numpy()


def dslash_bound(dims, kappa, bc_t, U, psi, sign):
    out, scale = dirac(dims, kappa, bc_t, U, psi, sign)
    return out, LD(2) ** -46.9 * scale[:, None] + LD(2) ** -52 * np.abs(out).reshape(-1, 12)


# tiles x columns above 152; a partial last tile, extents of 2, columns past one wave
@pytest.mark.parametrize("dims,cols", [((5, 3, 4, 7), 11), ((2, 2, 2, 40), 16), ((7, 3, 3, 5), 17), ((4, 4, 4, 4), 20)])
@pytest.mark.parametrize("kind,lk,kappa", [("gauss", "su3", 0.155), ("site_scales", "su3", -0.4),
                                           ("component_scales", "su3", 0.155), ("point", "unit", 0.125),
                                           ("sparse", "some_zero", 0.2), ("gauss", "general", 3e-4),
                                           ("gauss", "su3", 0.0), ("extreme", "su3", 0.155),
                                           ("gauss", "extreme", 0.155)])
def test_fixed_point_operator(seedlib, dims, cols, kind, lk, kappa):
    rng = np.random.default_rng(17)
    vol = int(np.prod(dims))
    for bc_t in (0, 1):
        x, U = blocks(kind, rng, vol, cols), links(lk, rng, dims)
        y = on_gpu(seedlib, dims, kappa, bc_t, U, x, 0)
        for j in (0, cols // 2, cols - 1):
            t, tau = dslash_bound(dims, kappa, bc_t, U, x[j], 1)
            ref, tol = dslash_bound(dims, kappa, bc_t, U, t, -1)
            tol = tol + 17 * dirac(dims, kappa, bc_t, U, tau.astype(CLD).ravel(), 1)[1][:, None]
            err = np.abs(y[j] - ref).reshape(vol, 12)
            assert np.all(err <= tol), (bc_t, j, float((err / tol).max()))


# tiles x columns up to 152, links and spinors converted in one launch: half a tile, a partial last one, several columns
@pytest.mark.parametrize("dims,cols", [((2, 2, 2, 2), 1), ((4, 4, 4, 4), 1), ((5, 3, 4, 7), 3), ((2, 3, 2, 5), 2)])
@pytest.mark.parametrize("kind,lk,kappa", [("gauss", "su3", 0.155), ("site_scales", "su3", -0.4),
                                           ("component_scales", "su3", 0.155), ("point", "unit", 0.125),
                                           ("sparse", "some_zero", 0.2), ("gauss", "general", 3e-4),
                                           ("gauss", "su3", 0.0), ("extreme", "su3", 0.155),
                                           ("gauss", "extreme", 0.155)])
def test_fixed_point_operator_few_sites(seedlib, dims, cols, kind, lk, kappa):
    test_fixed_point_operator(seedlib, dims, cols, kind, lk, kappa)


@pytest.mark.parametrize("dims,cols", [((4, 4, 4, 4), 20), ((6, 4, 5, 4), 12)])
def test_no_less_precise_than_fp64(seedlib, dims, cols):
    """D^H D on random spinors: error against extended precision no larger than the FP64 kernel's."""
    import torch
    rng = np.random.default_rng(5)
    vol, kappa = int(np.prod(dims)), 0.155
    x, U = blocks("gauss", rng, vol, cols), links("su3", rng, dims)
    y = on_gpu(seedlib, dims, kappa, 1, U, x, 0)
    X = torch.from_numpy(x).cuda().t()
    W = torch.empty_like(X.t()).t()
    seedlib.seed_wilson_apply_noalloc(dims, kappa, torch.from_numpy(U).cuda(), X, W, bc_t=1)
    w = W.t().cpu().numpy()
    for j in range(2):
        ref = dirac(dims, kappa, 1, U, dirac(dims, kappa, 1, U, x[j], 1)[0], -1)[0]
        e_fix, e_fp = (float(np.linalg.norm((v[j] - ref).astype(complex)) / np.linalg.norm(ref.astype(complex))) for v in (y, w))
        assert e_fix <= e_fp, (e_fix, e_fp)


def test_non_finite_values_as_in_fp64(seedlib):
    """Infinities and NaN spread to the same components as in the FP64 kernel."""
    import torch
    dims, kappa = (4, 3, 4, 4), 0.155
    rng = np.random.default_rng(6)
    vol = int(np.prod(dims))
    x, U = blocks("gauss", rng, vol, 32), links("su3", rng, dims)
    x[0, 12 * 7 + 2] = np.inf
    x[1, 12 * 100 + 4] = np.nan
    x[2, 12 * 9 + 11] = -1j * np.inf
    y = on_gpu(seedlib, dims, kappa, 0, U, x, 0)
    X = torch.from_numpy(x).cuda().t()
    W = torch.empty_like(X.t()).t()
    seedlib.seed_wilson_apply_noalloc(dims, kappa, torch.from_numpy(U).cuda(), X, W)
    w = W.t().cpu().numpy()
    assert np.array_equal(np.isfinite(y), np.isfinite(w))
    assert np.array_equal(np.isnan(y.real), np.isnan(w.real)) and np.array_equal(np.isnan(y.imag), np.isnan(w.imag))


def test_links_changed_in_place(seedlib):
    """The operator follows the caller's link array, as the FP64 kernel does."""
    import torch
    dims, kappa = (4, 4, 4, 4), 0.155
    rng = np.random.default_rng(7)
    x = blocks("gauss", rng, 256, 20)
    U1, U2 = links("su3", rng, dims), links("general", rng, dims)
    L = torch.from_numpy(U1).cuda()
    ctx = seedlib.seed_create_wilson(dims, kappa, L, seedlib.seed_params_default(m_max=2))
    X = torch.from_numpy(x).cuda().t()
    Y = torch.empty_like(X.t()).t()
    seedlib.seed_apply(ctx, 0, X, Y)
    L.copy_(torch.from_numpy(U2))
    seedlib.seed_apply(ctx, 0, X, Y)
    torch.cuda.synchronize()
    ref = on_gpu(seedlib, dims, kappa, 0, U2, x, 0)
    assert np.array_equal(Y.t().cpu().numpy(), ref)
    seedlib.seed_destroy(ctx)


def test_seed_steps_on_a_large_lattice(seedlib, orc):
    """From 16384 sites on the FP64 seed run takes step kernels with the fixed-point operator:
    D and D^H by themselves and the whole solve against the oracle, as in the parity tests."""
    from paper_0810_0330_gb300 import inputs as I
    from test_gpu_parity import REL_X, compare_full, dev_cols, host_cols, relerr, run_gpu, self_sensitivity, wilson_ctx
    import torch
    dims, kappa = (8, 16, 8, 16), 0.12
    U = I.random_su3_links(dims, 0.3, seed=2)
    B = I.gaussian_rhs(12 * 16384, 2, seed=3, complex_=True)
    kw = dict(m_max=200, reorth_freq=25)
    ctx = wilson_ctx(seedlib, dims, kappa, U, bc_t=1, tol_seed=1e-10, tol_rest=1e-8, **kw)
    for op_, sign in ((1, 1), (2, -1)):
        X = dev_cols(B)
        Y = torch.empty_like(X.t()).t()
        seedlib.seed_apply(ctx, op_, X, Y)
        ref = orc.wilson_dslash(dims, kappa, 1, sign, U, B[:, 1])
        assert relerr(host_cols(Y)[:, 1], ref) < 1e-15 * 4
    info1, info2, Xs, X = run_gpu(seedlib, ctx, B)
    op = orc.Operator.wilson(dims, kappa, U, bc_t=1)
    ref = orc.seed_solve_all(op, B, tol_seed=1e-10, tol_rest=1e-8, **kw)
    s_seed, s_final = self_sensitivity(orc, op, B, ref, cols=(1,), tol=1e-10, **kw)
    compare_full(ref, info1, info2, Xs, X, "wilson-large", seeded_tol=max(REL_X, 10 * s_seed),
                 final_tol=max(REL_X, 10 * s_final))
    seedlib.seed_destroy(ctx)


def test_fp32_operator_on_the_callers_layout_ragged(seedlib, orc):
    """FP32 operator from 65536 sites on (tiled through work space): a partial last
    tile and block, an odd column count, a leading dimension above n; the FP32 bound of test_gpu_mixed."""
    from paper_0810_0330_gb300 import inputs as I
    import torch
    dims, kappa = (17, 15, 17, 16), 0.155
    vol = int(np.prod(dims))
    n = 12 * vol
    rng = np.random.default_rng(4)
    U = I.random_su3_links(dims, 0.3, seed=5)
    ctx = seedlib.seed_create_wilson(dims, kappa, torch.from_numpy(U).cuda(),
                                     seedlib.seed_params_default(m_max=2, precision=1), bc_t=1)
    x = (rng.standard_normal((3, n + 5)) + 1j * rng.standard_normal((3, n + 5))).astype(np.complex64)
    buf = torch.from_numpy(x).cuda()
    for op, sign in ((3, 0), (4, 1), (5, -1)):
        y = torch.full((3, n + 7), 7.0, dtype=torch.complex64, device="cuda")
        seedlib.seed_apply(ctx, op, buf[:, :n].t(), y[:, :n].t())
        got = y.cpu().numpy()
        assert np.all(got[:, n:] == 7.0)   # nothing past the column's end
        v = x[2, :n].astype(np.complex128)
        if sign == 0:
            ref = orc.wilson_dslash(dims, kappa, 1, -1, U, orc.wilson_dslash(dims, kappa, 1, 1, U, v))
        else:
            ref = orc.wilson_dslash(dims, kappa, 1, sign, U, v)
        assert np.linalg.norm(got[2, :n] - ref) <= 1e-6 * np.linalg.norm(ref)
    seedlib.seed_destroy(ctx)


def test_apply_on_the_callers_stream(seedlib):
    """seed_apply runs on the context's stream: behind work queued there, and inside a capture
    whether the fixed-point work space is there (second round) or not (FP64 kernel).
    Bound: each form's D^H D is within 4e-15 of the exact one (9 terms of up to 8 roundings, twice)."""
    import torch
    dims, kappa = (4, 4, 4, 4), 0.155
    rng = np.random.default_rng(8)
    U = links("su3", rng, dims)
    x = blocks("gauss", rng, 256, 2)
    ref = on_gpu(seedlib, dims, kappa, 1, U, x, 0)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = seedlib.seed_create_wilson(dims, kappa, torch.from_numpy(U).cuda(), seedlib.seed_params_default(m_max=2),
                                         bc_t=1)
        src, X = torch.from_numpy(x).cuda(), torch.zeros(2, 3072, dtype=torch.complex128, device="cuda")
        Y = torch.zeros_like(X)
        seedlib.seed_apply(ctx, 1, X.t(), Y.t())   # work space for two columns
        for _ in range(2):
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                seedlib.seed_apply(ctx, 0, X.t(), Y.t())
            X.copy_(src)
            g.replay()
            got = Y.cpu().numpy()
            assert np.linalg.norm(got - ref) <= 8e-15 * np.linalg.norm(ref)
            X.zero_()
            torch.cuda._sleep(2000000)
            X.copy_(src)
            seedlib.seed_apply(ctx, 0, X.t(), Y.t())
            X.zero_()
            assert np.array_equal(Y.cpu().numpy(), ref)
    seedlib.seed_destroy(ctx)


@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 8])
def test_seeding_products_of_any_width(seedlib, orc, nrhs):
    """The block flush with 1, 2, 3, 4 and 4 + 3 seeded systems against the oracle; bounds as in
    the parity tests (the oracle's own sensitivity to a last-bit change)."""
    from paper_0810_0330_gb300 import inputs as I
    from test_gpu_parity import REL_X, compare_full, run_gpu, self_sensitivity, wilson_ctx
    dims, kappa = (3, 3, 5, 5), 0.13
    U = I.random_su3_links(dims, 0.3, seed=4)
    B = I.gaussian_rhs(12 * 225, nrhs, seed=5, complex_=True)
    kw = dict(m_max=300, reorth_freq=9)
    ctx = wilson_ctx(seedlib, dims, kappa, U, tol_seed=1e-10, tol_rest=1e-8, **kw)
    info1, info2, Xs, X = run_gpu(seedlib, ctx, B)
    op = orc.Operator.wilson(dims, kappa, U)
    ref = orc.seed_solve_all(op, B, tol_seed=1e-10, tol_rest=1e-8, **kw)
    s_seed, s_final = self_sensitivity(orc, op, B, ref, cols=(1,), tol=1e-10, **kw)
    compare_full(ref, info1, info2, Xs, X, "wilson-flush", seeded_tol=max(REL_X, 10 * s_seed),
                 final_tol=max(REL_X, 10 * s_final))
    seedlib.seed_destroy(ctx)
