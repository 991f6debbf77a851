"""stokes_precondition on uniform meshes with z over r, where S_hat^-1 allows it (degrees 0, 1 and 2 read each
entry of r_p only where they write it): the same result as beside it, and the identity rows hold r.

Tolerance: the same kernels on the same numbers, so FP64 1e-12 and FP32 2e-6 (the products' parity
bounds) for sums in any order; the identity rows are copies."""
import numpy as np
import pytest

import sinker_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels", [(3, 1), (12, 3)])
@pytest.mark.parametrize("schur_degree", [0, 1, 2])
@pytest.mark.parametrize("precond_kind", [0, 1])
def test_in_place(n, levels, schur_degree, precond_kind):
    import torch
    from paper_1907_06696_gb300 import capi
    o = capi.stokes_default_options()
    o.schur_degree, o.precond_kind = schur_degree, precond_kind
    prob = si.dr_problem(n, levels, 2, 1e3, 1949)
    ctx = capi.stokes_setup_problem(prob, options=o)
    M = 2 * n + 1
    inner = np.zeros((3, M, M, M), dtype=bool)
    inner[:, 1:-1, 1:-1, 1:-1] = True
    bnd = torch.tensor(~inner.ravel(), device="cuda")
    r = torch.tensor(si.uniform(51, ctx.n_u + ctx.n_p), device="cuda")
    for prec, tol in ((capi.STOKES_FP64, 1e-12), (capi.STOKES_FP32, 2e-6)):
        z = torch.full_like(r, 7.0)
        capi.stokes_precondition(ctx, prec, r, z)
        assert torch.equal(z[:ctx.n_u][bnd], r[:ctx.n_u][bnd])
        over = r.clone()
        capi.stokes_precondition(ctx, prec, over, over)
        assert torch.equal(over[:ctx.n_u][bnd], r[:ctx.n_u][bnd])
        assert float((over - z).norm()) <= tol * float(z.norm())
    ctx.close()
