"""A call whose work vectors are allocated on first use, after a first try that got some of them only (the
stokes_debug_alloc_limit hook lets the first so many bytes through): it gives ENOMEM then and works when the
memory is there. Each limit is what the vectors before the failing one take."""
import numpy as np
import pytest

import sinker_inputs as si

pytestmark = pytest.mark.gpu


def setup(capi, **options):
    o = capi.stokes_default_options()
    for k, v in options.items():
        setattr(o, k, v)
    prob = si.dr_problem(4, 2, 1, 1e2, 1953)
    return capi.stokes_setup_problem(prob, options=o)


def first_fails_then(capi, limit, call):
    lib = capi.load()
    assert lib.stokes_debug_alloc_limit(limit) == capi.STOKES_OK
    try:
        with pytest.raises(capi.StokesError) as e:
            call()
        assert e.value.status == capi.STOKES_ENOMEM
    finally:
        lib.stokes_debug_alloc_limit(-1)
    return call()


@pytest.mark.parametrize("vectors", [0, 1, 2])
def test_autotune(vectors):
    from paper_1907_06696_gb300 import capi
    ctx = setup(capi)
    block, _ = first_fails_then(capi, vectors * ctx.n_u * 4, lambda: capi.stokes_autotune(ctx, 1))
    assert block == 128
    ctx.close()


@pytest.mark.parametrize("vectors", [0, 3, 4, 6, 7])
def test_idr(vectors):
    import torch
    from paper_1907_06696_gb300 import capi
    ctx = setup(capi, outer_solver=1, idr_s=1)
    up = torch.zeros(ctx.n_u + ctx.n_p, dtype=torch.float64, device="cuda")
    info = first_fails_then(capi, vectors * (ctx.n_u + ctx.n_p) * 8,
                            lambda: capi.stokes_solve(ctx, capi.STOKES_FP64, None, up, rtol=1e-8, max_it=400))
    assert info.status == capi.STOKES_OK and info.rel_residual_true <= 1e-8
    ctx.close()


@pytest.mark.parametrize("vectors", [0, 1])
def test_solve_host(vectors):
    from paper_1907_06696_gb300 import capi
    ctx = setup(capi)
    rhs = np.concatenate([si.uniform(91, ctx.n_u), np.zeros(ctx.n_p)])
    up = np.zeros(ctx.n_u + ctx.n_p)
    info = first_fails_then(capi, vectors * (ctx.n_u + ctx.n_p) * 8,
                            lambda: capi.stokes_solve_host(ctx, capi.STOKES_FP64, rhs, up, rtol=1e-8, max_it=400))
    assert info.status == capi.STOKES_OK and np.isfinite(up).all()
    ctx.close()
