"""The fixed-point outer operator (csrc/outer.cuh) on small values: an operand times 2^k gives the result times 2^k as long
as both are normal FP64 numbers, also where a cell's largest exponent is too small for its zeros to fall out of the
rounding by themselves (fix_lift), and where the last scaling alone would be subnormal (fix_scale).

Host runs of the kernel's phases: bit for bit, every step before the last multiplication is the same integers. Compiled
kernels: 4e-15, the tolerance of the kernel's other tests (atomic adds come in any order)."""
import numpy as np
import pytest

from oracle import mesh
from test_outer_fixed import TOL, apply_host, rel, source, viscosity  # noqa: F401  (fixture)


@pytest.mark.parametrize("parts", ["up", "u", "p"])
@pytest.mark.parametrize("k", [-900, -945, -960, -980])
def test_small_values_scale_exactly(apply_host, k, parts):  # noqa: F811
    n = 3
    m = mesh.Mesh(n)
    mu = viscosity(n, 2)
    x = source(m, 1)
    if "u" not in parts:
        x[:m.n_u] = 0.0
    if "p" not in parts:
        x[m.n_u:] = 0.0
    du, dp = apply_host(n, mu, x)
    su, sp = apply_host(n, mu, np.ldexp(x, k))
    assert np.array_equal(su, np.ldexp(du, k)) and np.array_equal(sp, np.ldexp(dp, k))


@pytest.mark.gpu
@pytest.mark.parametrize("octree", [False, True])
def test_compiled_kernels_on_small_values(octree):
    import torch
    import sinker_inputs as si
    from paper_1907_06696_gb300 import capi
    ctx = capi.stokes_setup_octree_problem(si.octree_workload("oct_xs")) if octree else capi.stokes_setup_problem(si.workload("cube8"))
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand(ctx.n_u + ctx.n_p, generator=g, device="cuda", dtype=torch.float64) - 0.5
    scale = 2.0 ** -980
    for block, size, out in ((capi.BLOCK_STOKES, x.numel(), x.numel()), (capi.BLOCK_A, ctx.n_u, ctx.n_u), (capi.BLOCK_B, ctx.n_u, ctx.n_p)):
        src, one, small = x[:size].clone(), torch.empty(out, dtype=torch.float64, device="cuda"), torch.empty(out, dtype=torch.float64, device="cuda")
        capi.stokes_vmult(ctx, -1, block, capi.STOKES_FP64, src, one)
        capi.stokes_vmult(ctx, -1, block, capi.STOKES_FP64, src * scale, small)
        assert rel((small * 2.0 ** 500 * 2.0 ** 480).cpu().numpy(), one.cpu().numpy()) <= TOL
    ctx.close()
