"""The buffer of a plan's neighbour renders (8 bytes a pixel of every neighbour
patch) is there only where backgrounds are formed: not in a whole-field ELBO's
plans, beyond a 1,024th of the device's memory not before a plan's first
background, and once for all classes of a fit.  Taken while a stream is being
captured it gives the same values."""
import numpy as np
import pytest
import torch

from test_gpu_backgrounds import _scene

pytestmark = pytest.mark.gpu
N, SIDE = 24, 400
BUFFER = 8 * (N - 1) * SIDE * SIDE          # of one class: every source overlaps every other
# what a class's plan holds else: 8 bytes a pixel of background (1.3 MB), 256
# bytes a tile, tables of a few KB, in pages of 2 MB
PLANS = N * (4 << 20)
assert BUFFER + PLANS < N * BUFFER // 4


@pytest.fixture(scope="module")
def crowded():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = _scene(N, SIDE, 0)
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    plan = cel.Plan(ctx, dp, [0])           # kernels loaded, libraries initialised
    cel.background(plan), cel.render(plan), cel.elbo(plan)
    cel.FieldElbo(ctx, dp)()
    ctx.synchronize()
    del plan
    return cel, dp


def _taken(f):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    keep = f()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0], keep


def test_field_elbo_takes_none(crowded):
    cel, dp = crowded
    ctx = cel.Context(dp.host.model)        # a pool of its own
    taken, _ = _taken(lambda: cel.FieldElbo(ctx, dp))
    assert taken < PLANS + BUFFER


@pytest.fixture(scope="module")
def large(crowded):
    """Nine neighbours of 2,100 x 2,100 pixels: 318 MB."""
    cel, _ = crowded
    total = torch.cuda.mem_get_info()[1]
    side = 2100
    while 8 * 9 * side * side <= total // 1024:
        side += 100
    return cel, cel.DeviceProblem(_scene(10, side, 0)), 8 * 9 * side * side


def test_plan_takes_much_of_it_with_its_first_background(large):
    cel, dp, buffer = large
    ctx = cel.Context(dp.host.model)
    E = torch.zeros(2, dp.n_pool, dtype=torch.float32, device=ctx.device)

    def call(f, plan):
        cel._check(f(ctx.handle, plan.handle, cel._ptr(E[0]), cel._ptr(E[1])), "call")
        return plan

    # the plan's own: 8 bytes a pixel of one patch, a ninth
    taken, plan = _taken(lambda: call(cel.lib().celeste_render, cel.Plan(ctx, dp, [0])))
    assert taken < buffer // 2
    taken, _ = _taken(lambda: call(cel.lib().celeste_background, plan))
    assert buffer // 2 < taken < 2 * buffer
    assert _taken(lambda: call(cel.lib().celeste_background, plan))[0] == 0
    ctx.synchronize()


def test_plan_takes_little_of_it_at_once(crowded):
    cel, dp = crowded
    ctx = cel.Context(dp.host.model)
    taken, plan = _taken(lambda: cel.Plan(ctx, dp, [0]))
    assert taken >= BUFFER // 2
    E = torch.zeros(2, dp.n_pool, dtype=torch.float32, device=ctx.device)
    taken, _ = _taken(lambda: cel._check(cel.lib().celeste_background(
        ctx.handle, plan.handle, cel._ptr(E[0]), cel._ptr(E[1])), "b"))
    assert taken < BUFFER // 2
    ctx.synchronize()


def test_classes_of_a_fit_share_one(crowded):
    cel, dp = crowded
    ctx = cel.Context(dp.host.model)
    taken, fit = _taken(lambda: cel.Fit(ctx, dp, list(range(N))))
    assert fit.n_classes == N
    assert BUFFER // 2 < taken < PLANS + 2 * BUFFER


def test_first_background_under_capture(large):
    cel, dp, _ = large
    ref = [t.cpu().numpy() for t in cel.background(cel.Plan(cel.Context(dp.host.model), dp, [3, 4]))]
    side = torch.cuda.Stream()
    ctx = cel.Context(dp.host.model, stream=side)
    plan = cel.Plan(ctx, dp, [3, 4])
    E, V = (torch.zeros(dp.n_pool, dtype=torch.float32, device=ctx.device) for _ in range(2))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        cel._check(cel.lib().celeste_background(ctx.handle, plan.handle, cel._ptr(E), cel._ptr(V)), "b")
    for _ in range(2):
        E.zero_(), V.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(ref, (E, V)):
            assert np.array_equal(a, b.cpu().numpy())
    ctx.synchronize()
