"""Nothing that reaches a result is read before it is written: the STOKES_DEBUG build fills every device
allocation with NaN, and the calls whose work vectors are only partly written before their first use give
what the release build gives. Basis rows of odd length (n odd; octree meshes by chance) have one entry
past their end that no pass writes; a smoothing from a guess has no direction before it.

Tolerances: both builds run the same kernels, so solves agree to what their stopping test leaves (1e-9 of
the solution at rtol 1e-12 and 1e-6 at 1e-10 through contrasts of 1e4) with iteration counts within 2, and
the marching smoother, which has no atomic adds, bit for bit."""
import pytest

import sinker_inputs as si
from test_gpu_march import levels, vector

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def libs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_06696_gb300 import build as B
    from paper_1907_06696_gb300 import capi
    B.build()
    B.build(debug=True)
    capi.load()
    return capi, capi.open_library(capi.DEBUG_LIB_PATH)


def agree(capi, dbg, make, call, tol):
    ctx = make()
    want, its = call(ctx)
    ctx.close()
    with capi.use_library(dbg):
        ctx = make()
        got, its_d = call(ctx)
        ctx.close()
    assert torch.isfinite(got).all()
    assert float((got.double() - want.double()).norm()) <= tol * float(want.double().norm())
    assert abs(its - its_d) <= 2


def solver(capi, rtol):
    def call(ctx):
        N = ctx.n_u + ctx.n_p
        assert N % 2 == 1
        up = torch.zeros(N, dtype=torch.float64, device="cuda")
        info = capi.stokes_solve(ctx, capi.STOKES_FP32, None, up, rtol=rtol, max_it=400)
        assert info.status == capi.STOKES_OK
        return up, info.iterations
    return call


@pytest.mark.parametrize("n", [3, 5])
@pytest.mark.parametrize("gram_schmidt,outer_solver,restart", [(1, 0, 50), (0, 0, 50), (0, 2, 50), (1, 0, 5)])
def test_solve_with_basis_rows_of_odd_length(libs, n, gram_schmidt, outer_solver, restart):
    capi, dbg = libs
    prob = si.dr_problem(n, 1, 1, 1e2, 1943)

    def make():
        o = capi.stokes_default_options()
        o.gram_schmidt, o.outer_solver, o.restart = gram_schmidt, outer_solver, restart
        return capi.stokes_setup(prob.n, 1, prob.centres, prob.mu_min, prob.mu_max, options=o)
    agree(capi, dbg, make, solver(capi, 1e-12), 1e-9)


def test_octree_solve_with_basis_rows_of_odd_length(libs):
    capi, dbg = libs
    for seed in range(1945, 1985):
        prob = si.octree_problem(2, 2, 2, (4, 5), 1e4, seed, "odd")
        ctx = capi.stokes_setup_octree_problem(prob)
        odd = (ctx.n_u + ctx.n_p) % 2 == 1
        ctx.close()
        if odd:
            break
    assert odd
    agree(capi, dbg, lambda: capi.stokes_setup_octree_problem(prob), solver(capi, 1e-10), 1e-6)


@pytest.mark.parametrize("degree", [1, 2, 4])
def test_first_call_is_a_smoothing_from_a_guess(libs, degree):
    capi, dbg = libs
    n = 64
    M = 2 * n + 1
    inner = torch.zeros(3, M, M, M, device="cuda")
    inner[:, 1:-1, 1:-1, 1:-1] = 1

    def make():
        o = capi.stokes_default_options()
        o.cheb_degree = degree
        return capi.stokes_setup_problem(si.dr_problem(n, levels(n), 4, 1e4, 1947), options=o)

    def call(ctx):
        rhs, x = vector(torch, 41, ctx.n_u) * inner.view(-1), vector(torch, 42, ctx.n_u) * inner.view(-1)
        capi.stokes_smooth(ctx, ctx.n_levels - 1, capi.STOKES_FP32, rhs, x, 0)
        return x, 0
    agree(capi, dbg, make, call, 0.0)
