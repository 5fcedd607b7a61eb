"""Without a render cache a plan whose neighbours' overlaps cover at least half of
them (a quarter, with six neighbours on a pair) renders each neighbour pair
once and gathers its moments; below that every overlap is rendered.  Either
side of those lines, own patches of one pixel to several items, plans of some
of the sources only: the same bits as the gather from a render cache of every
source.  A Newton iteration renders the neighbours of the sources still
running only."""
import numpy as np
import pytest
import torch

from test_gpu_backgrounds import _scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,side,step,ppi,some", [
    (3, 1, 0, 256, False),     # one pixel
    (2, 16, 8, 256, False),    # a quarter, one neighbour: rendered over the overlaps
    (2, 24, 7, 256, False),    # 289 of 576: just above half
    (2, 24, 8, 256, False),    # 256 of 576: just below
    (86, 33, 24, 32, False),   # 3,010 items over small overlaps: four warps an item
    (100, 33, 24, 32, False),  # 3,500: a warp an item
    (4, 33, 1, 32, False),     # items of less than a row
    (9, 37, 2, 256, False),    # several items a neighbour, ragged
    (12, 33, 1, 1024, True),   # neighbours in and out of the plan
    (40, 70, 0, 256, True),    # more neighbours than lanes
])
def test_neighbours_rendered_once(n, side, step, ppi, some):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = _scene(n, side, step)
    ctx = cel.Context(p.model)
    ids = list(range(0, n, 3)) if some else list(range(n))
    got = []
    for cached in (False, True):
        dp = cel.DeviceProblem(p, render_cache=cached)
        if cached:
            cel.render_cache(cel.Plan(ctx, dp, list(range(n)), pixels_per_item=ppi))
        plan = cel.Plan(ctx, dp, ids, pixels_per_item=ppi)
        got.append([t.cpu().numpy() for t in cel.background(plan)])
    ctx.synchronize()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("stopped", [[], [0], [0, 2, 4], [1, 2, 3, 4, 5, 6], list(range(7))])
def test_newton_renders_for_running_sources(stopped):
    """With sources stopped (converged): the steps that the gather from a render
    cache gives, bit by bit, and nothing moved for the stopped ones."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = _scene(7, 33, 2)
    ctx = cel.Context(p.model)
    out = []
    for cached in (False, True):
        dp = cel.DeviceProblem(p, render_cache=cached)
        plan = cel.Plan(ctx, dp, list(range(7)))
        if cached:
            cel.render_cache(plan)
        start = dp.theta.clone()
        delta, status = cel.newton_state(dp)
        status[stopped] = 2
        cel.newton_step(plan, delta, status)
        assert torch.equal(dp.theta[stopped], start[stopped])
        out.append((dp.theta.cpu().numpy(), delta.cpu().numpy(), status.cpu().numpy()))
    ctx.synchronize()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
