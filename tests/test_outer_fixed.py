"""The fixed-point outer Stokes kernel (csrc/outer.cuh) where it can go wrong: a single cell and ragged
32-cell blocks, magnitudes far apart (within a cell, between velocity and pressure), zeros, values
at the ends of the FP64 range, NaN. Host runs of its phases (tests/native/outer_host.cpp) and the
compiled kernel, against the oracle in FP64.

Tolerance: the kernel rounds each input to 2^-55 of its cell's largest, and each result to 2^-53;
the oracle's own sums of up to 8 x 89 products are good to a few 2^-53. 4e-15 = 36 x 2^-53 in the
2-norm leaves both room; double-float pairs (6e-15) do not meet it."""
import ctypes as C

import numpy as np
import pytest

import sinker_inputs as si
from oracle import mesh, operators
from test_outer_host import host_build

TOL = 4e-15


@pytest.fixture(scope="module")
def apply_host(tmp_path_factory):
    L = host_build(tmp_path_factory, "outer_host.cpp")
    L.outer_apply_host.argtypes = [C.c_int] + [C.c_void_p] * 5

    def run(n, mu, x):
        m = mesh.Mesh(n)
        u, p = np.ascontiguousarray(x[:m.n_u]), np.ascontiguousarray(x[m.n_u:])
        du, dp = np.empty(m.n_u), np.empty(m.n_p)
        L.outer_apply_host(n, mu.ctypes.data, u.ctypes.data, p.ctypes.data, du.ctypes.data, dp.ctypes.data)
        return du, dp
    return run


def viscosity(n, decades, seed=71):
    return 10.0 ** si.uniform(seed, n ** 3, -decades, decades)


def source(m, decades, seed=73):
    x = si.uniform(seed, m.n_u + m.n_p)
    return x * 10.0 ** si.uniform(seed + 1, x.size, -decades, decades)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n,mu_decades,x_decades,p_scale", [
    (1, 0, 0, 1.0), (2, 3, 0, 1.0), (3, 3, 2, 1.0), (5, 2, 0, 1.0), (5, 12, 6, 1.0), (4, 1, 0, 2.0 ** 30), (4, 1, 0, 2.0 ** -40)])
def test_matches_oracle_to_fp64_rounding(apply_host, n, mu_decades, x_decades, p_scale):
    m = mesh.Mesh(n)
    mu = viscosity(n, mu_decades)
    x = source(m, x_decades)
    x[m.n_u:] *= p_scale
    ref = operators.Operators(m, mu).apply_stokes(x)
    du, dp = apply_host(n, mu, x)
    assert rel(du, ref[:m.n_u]) <= TOL
    assert rel(dp, ref[m.n_u:]) <= TOL


@pytest.mark.parametrize("k", [-700, -300, 300, 700])
def test_scaling_by_a_power_of_two_is_exact(apply_host, k):
    m = mesh.Mesh(3)
    mu = viscosity(3, 2)
    x = source(m, 1)
    du, dp = apply_host(3, mu, x)
    su, sp = apply_host(3, mu, np.ldexp(x, k))
    assert np.array_equal(su, np.ldexp(du, k)) and np.array_equal(sp, np.ldexp(dp, k))


def test_zero_and_rigid_fields(apply_host):
    m = mesh.Mesh(4)
    mu = viscosity(4, 3)
    du, dp = apply_host(4, mu, np.zeros(m.n_u + m.n_p))
    assert not du.any() and not dp.any()
    x = np.zeros(m.n_u + m.n_p)     # a constant pressure: B^T p = 0 on free rows up to rounding
    x[m.n_u:] = 3.0
    du, _ = apply_host(4, mu, x)
    assert np.abs(du).max() <= 1e-15 * 3.0 / 16


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_stays_in_its_cells(apply_host, bad):
    n = 4
    m = mesh.Mesh(n)
    mu = viscosity(n, 1)
    x = source(m, 0)
    M = 2 * n + 1
    node = 3 + M * (3 + M * 3)       # interior of cell (1, 1, 1)
    x[node] = bad
    du, dp = apply_host(n, mu, x)
    u = np.isfinite(du).reshape(3, M, M, M)
    assert not u[:, 2:5, 2:5, 2:5].any()
    u[:, 2:5, 2:5, 2:5] = True
    assert u.all()
    p = np.isfinite(dp).reshape(n + 1, n + 1, n + 1)
    assert not p[1:3, 1:3, 1:3].any()
    p[1:3, 1:3, 1:3] = True
    assert p.all()


@pytest.mark.gpu
@pytest.mark.parametrize("n,levels", [(2, 2), (3, 1), (5, 1), (8, 4), (12, 3)])
def test_compiled_kernel_matches_oracle_to_fp64_rounding(n, levels):
    import torch
    from paper_1907_06696_gb300 import capi
    m = mesh.Mesh(n)
    muq = np.repeat(viscosity(n, 3)[:, None], 27, axis=1)
    ctx = capi.stokes_setup(n, levels, mu_q=muq)
    ops = operators.Operators(m, muq[:, 0].copy())
    x = source(m, 1)
    src = torch.tensor(x, device="cuda")
    dst = torch.empty_like(src)
    capi.stokes_vmult(ctx, -1, capi.BLOCK_STOKES, capi.STOKES_FP64, src, dst)
    ref, got = ops.apply_stokes(x), dst.cpu().numpy()
    assert rel(got[:m.n_u], ref[:m.n_u]) <= TOL and rel(got[m.n_u:], ref[m.n_u:]) <= TOL
    du = torch.empty(m.n_u, dtype=torch.float64, device="cuda")
    capi.stokes_vmult(ctx, -1, capi.BLOCK_A, capi.STOKES_FP64, src[:m.n_u].clone(), du)
    assert rel(du.cpu().numpy(), ops.apply_A(x[:m.n_u])) <= TOL
    capi.stokes_vmult(ctx, -1, capi.BLOCK_B, capi.STOKES_FP64, src[:m.n_u].clone(), dst[:m.n_p])
    assert rel(dst[:m.n_p].cpu().numpy(), ref[m.n_u:]) <= TOL
    ctx.close()
