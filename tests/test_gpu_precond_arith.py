"""outer_arith = 0 asks for FP64 (or its accuracy) everywhere outside the V-cycle: the preconditioner's
r_u - B^T z_p too, also when the V-cycle is FP32. Double-float cannot hold |z_p| >= 2^128, FP64 can, and
B^T z_p is back inside the FP32 range: P^-1 is linear there as anywhere (S_hat = diag(M_p), which takes no
double-float of its own).

Tolerance: 2e-6, the FP32 products' parity bound, for sums in any order; the factor is a power of two."""
import numpy as np
import pytest

import sinker_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels", [(8, 4), (20, 3)])
def test_fp64_pressure_gradient_into_an_fp32_vcycle(n, levels):
    import torch
    from paper_1907_06696_gb300 import capi
    o = capi.stokes_default_options()
    o.outer_arith, o.schur_degree = 0, 0
    prob = si.dr_problem(n, levels, 1, 10.0, 1955)
    ctx = capi.stokes_setup(n, levels, prob.centres, 1e4 * prob.mu_min, 1e4 * prob.mu_max, options=o)
    r = np.concatenate([np.zeros(ctx.n_u), si.uniform(95, ctx.n_p)])
    z = torch.empty(r.size, dtype=torch.float64, device="cuda")
    capi.stokes_precondition(ctx, capi.STOKES_FP32, torch.tensor(r, device="cuda"), z)
    zp = z[ctx.n_u:].abs()
    k = 131 - int(torch.log2(zp.max()).ceil())          # the largest |z_p| in (2^130, 2^131]
    big = torch.empty_like(z)
    capi.stokes_precondition(ctx, capi.STOKES_FP32, torch.tensor(np.ldexp(r, k), device="cuda"), big)
    assert torch.isfinite(big).all()
    back = torch.ldexp(big, torch.tensor(-k, device="cuda"))
    assert float((back - z).norm()) <= 2e-6 * float(z.norm())
    assert float((back - z)[:ctx.n_u].norm()) <= 2e-6 * float(z[:ctx.n_u].norm())
    ctx.close()
