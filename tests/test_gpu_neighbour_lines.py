"""Where neighbours are rendered once each and where over every overlap: overlaps
of a half of the neighbours' pixels, 2^27 pixels, a quarter of the free
memory. The route shows in the number of launches; the values are the same
bits."""
import numpy as np
import pytest
import torch

from test_gpu_backgrounds import _scene

pytestmark = pytest.mark.gpu


def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    return cel


def _background(cel, ctx, plan, n):
    """E and V of the plan's first n pixels and the launches that formed them."""
    before = ctx.launches()
    E, V = cel.background(plan)
    return E[:n].clone(), V[:n].clone(), ctx.launches() - before


OVERLAPS, ONCE = 3, 4     # records, backgrounds (and renders), copy-out


@pytest.mark.parametrize("n,side,step,ids,route", [
    (7, 33, 7, [3], OVERLAPS),      # six neighbours, 0.361 of their pixels
    (7, 33, 9, [3], OVERLAPS),      # 0.256
    (6, 33, 5, [3], ONCE),          # five, 0.542
    (6, 33, 6, [3], OVERLAPS),      # 0.471
    (7, 33, 7, [0, 3], OVERLAPS),   # one of two pairs has six
    (9, 33, 3, [0, 3], ONCE),       # 0.877
])
def test_lines_of_the_overlap_rule(n, side, step, ids, route):
    cel = _setup()
    p = _scene(n, side, step)
    nb = [(s, t) for s in ids for t in range(n) if t != s and abs(t - s) * step < side]
    overlap = sum((side - abs(s - t) * step) ** 2 for s, t in nb)
    ratio = overlap / (len({t for _, t in nb}) * side * side)
    assert (route == ONCE) == (ratio >= 0.5)
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    E, V, launches = _background(cel, ctx, cel.Plan(ctx, dp, ids), dp.n_pool)
    assert launches == route
    dc = cel.DeviceProblem(p, render_cache=True)
    cel.render_cache(cel.Plan(ctx, dc, list(range(n))))
    Ec, Vc = cel.background(cel.Plan(ctx, dc, ids))
    ctx.synchronize()
    assert torch.equal(E, Ec) and torch.equal(V, Vc)


@pytest.fixture(scope="module")
def large():
    cel = _setup()
    p = _scene(33, 2048, 0)
    return cel, cel.DeviceProblem(p)


def test_renders_up_to_a_gigabyte(large):
    """32 neighbours of 2,048 x 2,048 pixels are 2^27; with a second source 33."""
    cel, dp = large
    ctx = cel.Context(dp.host.model)
    a = _background(cel, ctx, cel.Plan(ctx, dp, [0]), 2048 * 2048)
    b = _background(cel, ctx, cel.Plan(ctx, dp, [0, 1]), 2048 * 2048)
    ctx.synchronize()
    assert (a[2], b[2]) == (ONCE, OVERLAPS)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_no_more_than_a_quarter_of_the_free_memory(large):
    """With 3.5 GB free, 1 GB is not taken; the overlaps give the same values,
    and the plan stays with them."""
    cel, dp = large
    ctx = cel.Context(dp.host.model)
    a = _background(cel, ctx, cel.Plan(ctx, dp, [0]), 2048 * 2048)
    ctx.synchronize()
    ctx = cel.Context(dp.host.model)               # (without the block that the other one keeps)
    plan = cel.Plan(ctx, dp, [0])
    torch.cuda.empty_cache()
    E = torch.zeros(2, dp.n_pool, dtype=torch.float32, device=ctx.device)
    torch.cuda.synchronize()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (3500 << 20), dtype=torch.uint8, device=ctx.device)
    counts = []
    for _ in range(2):
        before = ctx.launches()
        cel._check(cel.lib().celeste_background(ctx.handle, plan.handle, cel._ptr(E[0]), cel._ptr(E[1])), "b")
        ctx.synchronize()
        counts.append(ctx.launches() - before)
        if fill is not None:
            fill = None
            torch.cuda.empty_cache()
    assert counts == [OVERLAPS, OVERLAPS]
    n = 2048 * 2048
    assert torch.equal(E[0, :n], a[0]) and torch.equal(E[1, :n], a[1])
