"""Smoothing from a guess does not depend on what an earlier call left in the level's work vectors: after a call
whose right-hand side or guess held a NaN or an infinity, finite data give what a fresh context gives. One
size of every FP32 level operator: blocks (16), cells (24), marching tiles (64, where vectors off a 16-byte
boundary take the cells).

Tolerance: the operators without atomic adds repeat bit for bit; the cell operator's sums of up to 8 cells
come in any order, 2e-6 (the FP32 product's parity bound)."""
import numpy as np
import pytest

import sinker_inputs as si
from test_gpu_march import levels, vector

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("n", [16, 24, 64])
def test_a_guess_after_non_finite_data(n, bad):
    import torch
    from paper_1907_06696_gb300 import capi
    prob = si.dr_problem(n, levels(n), 4, 1e4, 1933)
    used, fresh = capi.stokes_setup_problem(prob), capi.stokes_setup_problem(prob)
    M = 2 * n + 1
    inner = torch.zeros(3, M, M, M, device="cuda")
    inner[:, 1:-1, 1:-1, 1:-1] = 1
    rhs, x0 = vector(torch, 31, used.n_u) * inner.view(-1), vector(torch, 32, used.n_u) * inner.view(-1)
    spoilt = rhs.clone().view(3, M, M, M)
    spoilt[:, M // 2, M // 2, M // 2] = bad
    x = x0.clone()
    capi.stokes_smooth(used, used.n_levels - 1, capi.STOKES_FP32, spoilt.view(-1), x, 0)
    assert not torch.isfinite(x).all()
    for zero_guess in (0, 1):
        x, ref = x0.clone(), x0.clone()
        capi.stokes_smooth(used, used.n_levels - 1, capi.STOKES_FP32, rhs, x, zero_guess)
        capi.stokes_smooth(fresh, fresh.n_levels - 1, capi.STOKES_FP32, rhs, ref, zero_guess)
        assert torch.isfinite(x).all()
        assert float((x.double() - ref.double()).norm()) <= (2e-6 if n == 24 else 0.0) * float(ref.double().norm())
    used.close()
    fresh.close()
