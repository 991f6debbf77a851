"""The marching FP32 level operator (csrc/march.cu): products, residuals and Chebyshev steps at its
smallest size and at sizes whose tiles and layer chunks end ragged, against the component-split
operator with separate vector passes (vmult_kernel = 3, itself checked against the oracle).

Tolerance 2e-5, the FP32 smoothing bound of the parity tests: both sides round the same FP32 inputs
and differ in the order of sums of up to 8 cells and in where the vector update rounds."""
import numpy as np
import pytest

import sinker_inputs as si

pytestmark = pytest.mark.gpu
TOL = 2e-5


def levels(n):
    k = 1
    while n % 2 == 0:
        n, k = n // 2, k + 1
    return k


def make(capi, n, kernel, degree=4):
    o = capi.stokes_default_options()
    o.vmult_kernel, o.cheb_degree = kernel, degree
    return capi.stokes_setup_problem(si.dr_problem(n, levels(n), 4, 1e4, 1931), options=o)


def vector(torch, seed, n):
    return torch.tensor(si.uniform(seed, n).astype(np.float32), device="cuda")


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("n", [64, 80, 96, 160])
def test_products_and_vcycle_match_the_split_operator(n):
    import torch
    from paper_1907_06696_gb300 import capi
    a, b = make(capi, n, 0), make(capi, n, 3)
    src = vector(torch, 11, a.n_u)
    da, db = torch.full_like(src, 7.0), torch.empty_like(src)
    capi.stokes_vmult(a, -1, capi.BLOCK_A, capi.STOKES_FP32, src, da)
    capi.stokes_vmult(b, -1, capi.BLOCK_A, capi.STOKES_FP32, src, db)
    assert rel(da, db) <= 2e-6
    buf = torch.empty(a.n_u + 4, device="cuda")          # views off a 16-byte boundary take the cell kernel
    view = buf[1:1 + a.n_u]
    capi.stokes_vmult(a, -1, capi.BLOCK_A, capi.STOKES_FP32, src, view)
    assert rel(view, db) <= 2e-6
    for _ in range(2):                                   # the second cycle finds the first one's buffers
        capi.gmg_vcycle(a, capi.STOKES_FP32, src, da)
    capi.gmg_vcycle(b, capi.STOKES_FP32, src, db)
    assert rel(da, db) <= TOL
    a.close()
    b.close()


@pytest.mark.parametrize("degree", [1, 2, 3, 4])
@pytest.mark.parametrize("zero_guess", [0, 1])
def test_smoothing_of_every_parity(degree, zero_guess):
    """The iterates alternate between two buffers; odd and even step counts end in the caller's."""
    import torch
    from paper_1907_06696_gb300 import capi
    n = 64
    a, b = make(capi, n, 0, degree), make(capi, n, 3, degree)
    rhs, x0 = vector(torch, 21, a.n_u), vector(torch, 22, a.n_u)
    M = 2 * n + 1
    inner = torch.zeros(3, M, M, M, device="cuda")
    inner[:, 1:-1, 1:-1, 1:-1] = 1
    rhs, x0 = rhs * inner.view(-1), x0 * inner.view(-1)
    xa, xb = x0.clone(), x0.clone()
    for _ in range(2):
        capi.stokes_smooth(a, a.n_levels - 1, capi.STOKES_FP32, rhs, xa, zero_guess)
        capi.stokes_smooth(b, b.n_levels - 1, capi.STOKES_FP32, rhs, xb, zero_guess)
    assert rel(xa, xb) <= TOL
    assert not (xa * (1 - inner.view(-1))).any()
    a.close()
    b.close()
