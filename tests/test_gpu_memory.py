"""Work space of the fixed-point Wilson operator is optional: where the device has no room for
it, every call still runs, in FP64 arithmetic, and takes it up again once there is room."""
import numpy as np
import pytest

from paper_0810_0330_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS, KAPPA, COLS = (16, 16, 16, 16), 0.10, 12
N = 12 * I.lattice_sites(DIMS)
BLOCK = 16 * N * COLS   # bytes of a block of FP64 columns: 151 MB


def fill(leave):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def fp64_normal(seedlib, U, X, W, Y):
    """Graph of Y = D^H (W = D X) in FP64 arithmetic: the captured forms, which take no work space."""
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        ctx = seedlib.seed_create_wilson(DIMS, KAPPA, U, seedlib.seed_params_default(m_max=2), bc_t=1)
        seedlib.seed_apply(ctx, 1, X, W)   # room for the columns
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            seedlib.seed_apply(ctx, 1, X, W)
            seedlib.seed_apply(ctx, 2, W, Y)
    torch.cuda.synchronize()
    return ctx, graph


@pytest.mark.parametrize("precision", [0, 1])
def test_calls_run_without_room_for_the_fixed_point_form(seedlib, precision):
    g = torch.Generator("cuda").manual_seed(1)
    B = torch.randn(COLS, N, dtype=torch.complex128, device="cuda", generator=g).t()
    U = torch.from_numpy(I.random_su3_links(DIMS, 0.3, seed=5)).cuda()
    X, Y, W, A, V = (torch.zeros(COLS, N, dtype=torch.complex128, device="cuda").t() for _ in range(5))
    prm = dict(m_max=300, tol_seed=1e-8, tol_rest=1e-8, precision=precision)
    torch.cuda.synchronize()
    ref, normal = fp64_normal(seedlib, U, V, W, A)   # A = D^H D V
    V.copy_(B)
    normal.replay()
    want = A.clone()
    ctx = seedlib.seed_create_wilson(DIMS, KAPPA, U, seedlib.seed_params_default(**prm), bc_t=1)
    # room for the columns every call needs (FP64: four blocks; mixed: FP32 ones too), not for a fifth
    need = 4 * BLOCK + (5 * BLOCK // 2 + BLOCK // COLS // 2 if precision else 0)
    full = fill(need + 2 * BLOCK // 3)
    seedlib.seed_apply(ctx, 0, B, Y)
    torch.cuda.synchronize()
    assert torch.equal(Y, want)   # the FP64 kernels' bits
    for again in range(2):   # without room, then with it
        X.zero_()
        info = seedlib.seed_solve_cg(ctx, B, X)
        V.copy_(X)
        normal.replay()
        A.sub_(B)
        assert all(i["converged"] == 1 for i in info)
        for j in range(COLS):
            assert float(torch.linalg.vector_norm(A[:, j])) <= 1.01e-8 * float(torch.linalg.vector_norm(B[:, j]))
        info = seedlib.seed_solve_first(ctx, B[:, :1], X[:, :1])
        assert info[0]["converged"] == 1
        if again == 0:
            del full
            torch.cuda.empty_cache()
    seedlib.seed_apply(ctx, 0, B, Y)
    torch.cuda.synchronize()
    assert not torch.equal(Y, want)   # the fixed-point form again ...
    fresh = seedlib.seed_create_wilson(DIMS, KAPPA, U, seedlib.seed_params_default(**prm), bc_t=1)
    seedlib.seed_apply(fresh, 0, B, A)
    torch.cuda.synchronize()
    assert torch.equal(Y, A)      # ... with a fresh context's bits
    for c in (fresh, ctx, ref):
        seedlib.seed_destroy(c)


def test_first_captured_application_has_the_later_ones_bits(seedlib):
    """A context's first application of A is a captured one, or not: the same bits."""
    dims = (4, 4, 4, 4)
    U = torch.from_numpy(I.random_su3_links(dims, 0.3, seed=5)).cuda()
    g = torch.Generator("cuda").manual_seed(1)
    out = []
    for captured in (False, True):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            X = torch.randn(2, 3072, dtype=torch.complex128, device="cuda", generator=g.manual_seed(2)).t()
            Y = torch.zeros_like(X.t()).t()
            ctx = seedlib.seed_create_wilson(dims, 0.155, U, seedlib.seed_params_default(m_max=2))
            seedlib.seed_apply(ctx, 1, X, Y)   # room for two columns, none for the fixed-point form
            s.synchronize()
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    seedlib.seed_apply(ctx, 0, X, Y)
                graph.replay()
            else:
                seedlib.seed_apply(ctx, 0, X, Y)
            s.synchronize()
        out.append(Y.clone())
        seedlib.seed_destroy(ctx)
    assert torch.equal(out[0], out[1])
