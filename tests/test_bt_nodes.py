"""B^T p gathered per cell (csrc/pressure.cuh bt_nodes) against the oracle's element-assembled B^T: one
cell (no neighbour on any side), odd and even sizes, pressures over 12 decades.

Tolerance: a node sums at most 8 values of one sign pattern, so FP64 is good to 16 x 2^-53 = 1.8e-15 of the
values' size and double-float (2^-47 per operation, 8 operations) to 5.7e-14; the 2-norm bounds 2e-15 and
2e-13 leave room for the oracle's own rounding."""
import ctypes as C

import numpy as np
import pytest

import sinker_inputs as si
from oracle import mesh, operators
from test_outer_host import host_build


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    L = host_build(tmp_path_factory, "bt_nodes_host.cpp")
    for f in (L.bt_nodes_f64, L.bt_nodes_df64):
        f.restype, f.argtypes = None, [C.c_int, C.c_void_p, C.c_void_p]
    return L


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("decades", [0, 6])
def test_matches_oracle(lib, n, decades):
    m = mesh.Mesh(n)
    p = si.uniform(81, m.n_p) * 10.0 ** si.uniform(82, m.n_p, -decades, decades)
    ops = operators.Operators(m, np.ones(n ** 3))
    ref = ops.apply_stokes(np.concatenate([np.zeros(m.n_u), p]))[:m.n_u]
    for f, tol in ((lib.bt_nodes_f64, 2e-15), (lib.bt_nodes_df64, 2e-13)):
        out = np.empty(m.n_u)
        f(n, p.ctypes.data, out.ctypes.data)
        assert np.linalg.norm(out - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.gpu
@pytest.mark.parametrize("n,levels", [(2, 2), (3, 1), (5, 1), (8, 4), (12, 3)])
def test_block_and_preconditioner(n, levels):
    """The B^T block, and the preconditioner's right-hand side through P^-1 in both precisions."""
    import torch
    from oracle import gmg, krylov, sinker
    from paper_1907_06696_gb300 import capi
    prob = si.dr_problem(n, levels, 2, 1e2, 1951)
    ctx = capi.stokes_setup_problem(prob)
    m = mesh.Mesh(n)
    mus = sinker.level_viscosities(m, prob, levels)
    ops = operators.Operators(m, mus[-1])
    p = si.uniform(83, m.n_p)
    out = torch.full((m.n_u,), 7.0, dtype=torch.float64, device="cuda")
    capi.stokes_vmult(ctx, -1, capi.BLOCK_BT, capi.STOKES_FP64, torch.tensor(p, device="cuda"), out)
    ref = ops.apply_stokes(np.concatenate([np.zeros(m.n_u), p]))[:m.n_u]
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 2e-15 * np.linalg.norm(ref)
    r = si.uniform(84, m.n_u + m.n_p)
    z = torch.full((m.n_u + m.n_p,), 7.0, dtype=torch.float64, device="cuda")
    ref = krylov.StokesPreconditioner(ops, gmg.GMG(n, levels, mus)).apply(r)
    for prec, tol in ((capi.STOKES_FP64, 1e-10), (capi.STOKES_FP32, 2e-5)):   # the parity bounds of the V-cycles
        for _ in range(2):
            capi.stokes_precondition(ctx, prec, torch.tensor(r, device="cuda"), z)
            assert np.linalg.norm(z.cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    ctx.close()
