"""The block-size tuner works where the cell operator runs: on the finest level of 17 to 63 cells per axis, also
when the finest level of all takes another operator, and its candidates hold the untuned size. Seen from
outside: the products it launches, the size it returns, the product and the V-cycle's time afterwards.

Each of the four candidates takes 4 x 10 products of at least one launch. The products agree to 2e-6, the FP32
parity bound; the V-cycle may take 1.1 times the untuned time, medians of 21, far above the noise of either."""
import pytest

import sinker_inputs as si
from test_gpu_march import levels, rel, vector

pytestmark = pytest.mark.gpu


def vcycle_us(capi, torch, ctx, src, dst):
    times = []
    for _ in range(24):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            capi.gmg_vcycle(ctx, capi.STOKES_FP32, src, dst)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 200.0)
    return sorted(times[3:])[10]


@pytest.mark.parametrize("n,tunes", [(16, False), (20, True), (24, True), (40, True), (64, True), (80, True)])
def test_tunes_the_level_that_takes_the_cell_operator(n, tunes):
    import torch
    from paper_1907_06696_gb300 import capi
    ctx = capi.stokes_setup_problem(si.dr_problem(n, levels(n), 4, 1e4, 1951))
    src = vector(torch, 61, ctx.n_u)
    before, after = torch.empty_like(src), torch.empty_like(src)
    capi.stokes_vmult(ctx, -1, capi.BLOCK_A, capi.STOKES_FP32, src, before)
    untuned = vcycle_us(capi, torch, ctx, src, after)
    count = capi.stokes_launch_count()
    block, _ = capi.stokes_autotune(ctx, 1)
    count = capi.stokes_launch_count() - count
    assert count >= 160 if tunes else count < 10
    assert block in ((32, 64, 128, 256) if tunes else (128,))
    capi.stokes_vmult(ctx, -1, capi.BLOCK_A, capi.STOKES_FP32, src, after)
    assert rel(after, before) <= 2e-6
    assert vcycle_us(capi, torch, ctx, src, after) <= 1.1 * untuned
    assert capi.stokes_autotune(ctx, 2)[0] == block        # the degree alone leaves the block size
    ctx.close()
