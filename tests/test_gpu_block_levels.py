"""The FP32 operator of the small levels (csrc/block.cu): products, smoothing steps and V-cycles against the
component-split operator with separate vector passes (vmult_kernel = 3, itself checked against the
oracle): one cell, sizes that end inside a block, every coarsest mesh, every parity of the Chebyshev
degree from zero and from a guess; V-cycles twice, since the first leaves its buffers to the second.

Tolerances: 2e-6 for a product and 2e-5 for smoothing and the V-cycle, the FP32 bounds of the parity tests:
the same steps with the sums of up to 8 cells in another order."""
import numpy as np
import pytest

import sinker_inputs as si

pytestmark = pytest.mark.gpu


def make(capi, n, levels, kernel, degree=4):
    o = capi.stokes_default_options()
    o.vmult_kernel, o.cheb_degree = kernel, degree
    return capi.stokes_setup_problem(si.dr_problem(n, levels, 3, 1e3, 1961), options=o)


def vector(torch, seed, n):
    return torch.tensor(si.uniform(seed, n).astype(np.float32), device="cuda")


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("n,levels", [(1, 1), (2, 1), (3, 1), (5, 1), (6, 1), (10, 2), (12, 3), (20, 3), (40, 4)])
def test_product(n, levels):
    import torch
    from paper_1907_06696_gb300 import capi
    a, b = make(capi, n, levels, 0), make(capi, n, levels, 3)
    src = vector(torch, 31, a.n_u)
    buf, ref = torch.full((a.n_u + 3,), 7.0, device="cuda"), torch.empty_like(src)
    capi.stokes_vmult(b, -1, capi.BLOCK_A, capi.STOKES_FP32, src, ref)
    for off in (0, 1, 2):       # views at any 4-byte offset
        out = buf[off:off + a.n_u]
        capi.stokes_vmult(a, -1, capi.BLOCK_A, capi.STOKES_FP32, src, out)
        assert rel(out, ref) <= 2e-6
    a.close()
    b.close()


@pytest.mark.parametrize("degree", [1, 2, 3, 4])
@pytest.mark.parametrize("zero_guess", [0, 1])
@pytest.mark.parametrize("n,levels", [(2, 2), (12, 3)])
def test_smoothing(degree, zero_guess, n, levels):
    import torch
    from paper_1907_06696_gb300 import capi
    a, b = make(capi, n, levels, 0, degree), make(capi, n, levels, 3, degree)
    M = 2 * n + 1
    inner = torch.zeros(3, M, M, M, device="cuda")
    inner[:, 1:-1, 1:-1, 1:-1] = 1
    inner = inner.view(-1)
    rhs, x0 = vector(torch, 41, a.n_u) * inner, vector(torch, 42, a.n_u) * inner
    xa, xb = x0.clone() + (7.0 * (1 - inner) if zero_guess else 0), x0.clone()
    for _ in range(2):
        capi.stokes_smooth(a, a.n_levels - 1, capi.STOKES_FP32, rhs, xa, zero_guess)
        capi.stokes_smooth(b, b.n_levels - 1, capi.STOKES_FP32, rhs, xb, zero_guess)
    assert rel(xa, xb) <= 2e-5
    assert not (xa * (1 - inner)).any()
    a.close()
    b.close()


@pytest.mark.parametrize("n,levels,degree", [
    (1, 1, 4), (2, 2, 4), (4, 2, 4), (4, 3, 1), (8, 4, 2), (16, 5, 4), (16, 5, 3), (32, 6, 4), (6, 2, 5), (12, 3, 4),
    (12, 2, 8), (8, 2, 4), (16, 3, 4), (10, 2, 4), (20, 3, 4), (24, 4, 4), (12, 3, 9), (48, 5, 4)])
def test_vcycle(n, levels, degree):
    import torch
    from paper_1907_06696_gb300 import capi
    a, b = make(capi, n, levels, 0, degree), make(capi, n, levels, 3, degree)
    src = vector(torch, 51, a.n_u)
    ref, got = torch.empty_like(src), [torch.full_like(src, 7.0) for _ in range(2)]
    capi.gmg_vcycle(b, capi.STOKES_FP32, src, ref)
    for g in got:
        capi.gmg_vcycle(a, capi.STOKES_FP32, src, g)
        assert rel(g, ref) <= 2e-5
    assert rel(got[0], got[1]) <= 2e-6
    a.close()
    b.close()
