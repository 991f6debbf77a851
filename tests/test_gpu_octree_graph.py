"""The captured V-cycle of octree meshes against the same launches one by one (graphs = 0): right-hand side
and result in new buffers on each call, an in-place call, and a caller that captures its own stream.

The two differ by the order of the atomic additions only: FP64 1e-12; FP32 1e-5 (a few roundings of
6e-8 per smoothing step, carried through some 50 steps).
"""
import pytest

import sinker_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_06696_gb300 import build as B
    from paper_1907_06696_gb300 import capi as api
    B.build()
    api.load()
    return api


def rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("precond", [0, 1])
def test_graph_matches_launches(capi, prec, precond):
    pr, tol = (capi.STOKES_FP64, 1e-12) if prec == "fp64" else (capi.STOKES_FP32, 1e-5)
    p = si.octree_workload("oct_s")
    ctxs = []
    for graphs in (0, 1):
        o = capi.stokes_default_options()
        o.graphs, o.precond_kind = graphs, precond
        ctxs.append(capi.stokes_setup_octree_problem(p, options=o))
    n, m = ctxs[0].n_u, ctxs[0].n_p
    gen = torch.Generator().manual_seed(7)
    for k in range(3):
        b = torch.randn(n + m, generator=gen, dtype=torch.float64).cuda()
        ref, got = torch.empty_like(b), torch.empty_like(b)
        capi.stokes_precondition(ctxs[0], pr, b, ref)
        capi.stokes_precondition(ctxs[1], pr, b, got)
        assert rel(got, ref) <= tol, k
        bu = b[:n].clone()
        x, y = torch.empty_like(bu), bu.clone()
        capi.gmg_vcycle(ctxs[0], pr, bu, x)
        capi.gmg_vcycle(ctxs[1], pr, y, y)
        assert rel(y, x) <= tol, k
    for c in ctxs:
        c.close()


def test_caller_captures(capi):
    ctx = capi.stokes_setup_octree_problem(si.octree_workload("oct_s"))
    gen = torch.Generator().manual_seed(8)
    b = torch.randn(ctx.n_u, generator=gen, dtype=torch.float64).cuda()
    x, ref = torch.empty_like(b), torch.empty_like(b)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        capi.gmg_vcycle(ctx, capi.STOKES_FP64, b, x, stream=s.cuda_stream)
        s.synchronize()
        g.capture_begin()
        capi.gmg_vcycle(ctx, capi.STOKES_FP64, b, x, stream=s.cuda_stream)
        g.capture_end()
    for k in range(2):
        b.copy_(torch.randn(ctx.n_u, generator=gen, dtype=torch.float64))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        capi.gmg_vcycle(ctx, capi.STOKES_FP64, b, ref)
        torch.cuda.synchronize()
        assert rel(x, ref) <= 1e-12, k
    ctx.close()
