"""Pressures whose size against the viscosity takes the fixed-point scale of the outer Stokes kernel
(csrc/outer.cuh fix_scale) out of the FP64 exponent range although the result is well inside: B^T p does not
depend on the viscosity. Host runs of the kernel's phases; u zero, and u whose A u is below the last bit of B^T p.

Tolerance: that of the kernel's other tests, an exact power of two apart."""
import numpy as np
import pytest

import sinker_inputs as si
from oracle import mesh, operators
from test_outer_fixed import TOL, apply_host, rel, viscosity  # noqa: F401  (fixture)


@pytest.mark.parametrize("k,mu_exp,u_exp", [
    (0, 0, None), (-940, 40, None), (-940, 60, None), (-940, 300, None), (900, -100, None), (900, -200, None),
    (900, -600, None), (900, -200, -1000), (900, -200, -1060), (0, -300, -960)])
def test_pressure_gradient_at_any_viscosity(apply_host, k, mu_exp, u_exp):  # noqa: F811
    n = 3
    m = mesh.Mesh(n)
    mu = viscosity(n, 1)
    p = si.uniform(77, m.n_p)
    x = np.zeros(m.n_u + m.n_p)
    x[m.n_u:] = p
    ref = operators.Operators(m, mu).apply_stokes(x)[:m.n_u]
    x[m.n_u:] = np.ldexp(p, k)
    if u_exp is not None:
        x[:m.n_u] = np.ldexp(si.uniform(78, m.n_u), u_exp)
    du, _ = apply_host(n, np.ldexp(mu, mu_exp), x)
    M = 2 * n + 1
    inner = np.zeros((3, M, M, M), dtype=bool)
    inner[:, 1:-1, 1:-1, 1:-1] = True
    inner = inner.ravel()
    assert rel(np.ldexp(du[inner], -k), ref[inner]) <= TOL
