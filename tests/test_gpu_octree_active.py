"""Octree operators at the edges of their blocks, against the CPU oracle (oracle/adaptive.py): meshes with fewer
leaves than a block of 32, without hanging nodes, with a last block that is partly filled, and with
more blocks than SMs; the V-cycle on
hierarchies of two to five levels.

Tolerances as in test_gpu_octree.py: blocks 1e-12 (same sums, another order), V-cycle FP64 1e-9, FP32 1e-4.
"""
import numpy as np
import pytest

import sinker_inputs as si
from oracle import adaptive, octree

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# base level, coarsest level, sinkers, their levels
MESHES = [(1, 1, 1, (2,)), (1, 1, 1, (3,)), (2, 1, 1, (2,)), (2, 2, 3, (3, 4)), (2, 1, 2, (5,)), (4, 2, 1, (6,))]


@pytest.fixture(scope="module")
def capi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_06696_gb300 import build as B
    from paper_1907_06696_gb300 import capi as api
    B.build()
    api.load()
    return api


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(device="cuda", dtype=torch.float64)


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("mesh", MESHES)
def test_blocks_and_vcycle(capi, mesh):
    base, coarsest, sinkers, levels = mesh
    p = si.octree_problem(base, coarsest, sinkers, levels, 1e3, 1941)
    t = octree.Octree(octree.balance(octree.refine_shells(p.base_level, p.centres, p.max_levels, p.shell_radius,
                                                          p.shell_half_width)), p.coarsest_level)
    S = adaptive.AdaptiveStokes(t, p)
    ctx = capi.stokes_setup_octree_problem(p)
    u, q = si.uniform(3301, S.n_u), si.uniform(3302, S.n_p)
    up = np.concatenate([u, q])
    for blk, src, ref in [(capi.BLOCK_A, u, S.apply_A(u)), (capi.BLOCK_B, u, S.apply_B(u)), (capi.BLOCK_BT, q, S.apply_BT(q)),
                          (capi.BLOCK_MP, q, S.apply_Mp(q)), (capi.BLOCK_STOKES, up, S.apply_stokes(up))]:
        out = torch.empty(ref.size, dtype=torch.float64, device="cuda")
        capi.stokes_vmult(ctx, -1, blk, capi.STOKES_FP64, dev(src), out)
        assert rel(out, ref) <= 1e-12, blk
    ref = S.vcycle(u)
    for prec, tol in ((capi.STOKES_FP64, 1e-9), (capi.STOKES_FP32, 1e-4)):
        x = torch.empty(S.n_u, dtype=torch.float64, device="cuda")
        capi.gmg_vcycle(ctx, prec, dev(u), x)
        assert rel(x, ref) <= tol, prec
    ctx.close()
