"""Launches of few items take a block per item (derivative and value passes);
they give the bits of the persistent kernels, which larger plans of the same
sources take."""
import numpy as np
import pytest
import torch

import fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,ppi", [(15, 256), (17, 256), (16, 32), (33, 96), (41, 256), (41, 1024)])
def test_block_per_item_equals_persistent_bitwise(side, ppi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    # ragged: 225 and 289 pixels, one pass, 96-pixel items, one item of seven
    # passes, items longer than a block
    p = fields.batched(seed=70, n_sources=280, min_side=side, max_side=side, max_images_per_band=2,
                       max_neighbours=2)
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    items = p.n_patches * -(-side * side // ppi)
    assert items > 8 * n_sm, "the large plan takes the persistent kernels"
    big = cel.Plan(ctx, dp, list(range(p.n_sources)), pixels_per_item=ppi)
    ref = [t.cpu().numpy() for t in cel.elbo_grad_hess(big)]
    val = [t.cpu().numpy() for t in cel.elbo(big)]
    delta, status = cel.newton_state(dp)
    theta0 = dp.theta.clone()
    cel.newton_step(big, delta, status)
    theta, st = dp.theta.cpu().numpy(), status.cpu().numpy()
    for s in (0, 137, 279):
        dp.theta.copy_(theta0)
        one = cel.Plan(ctx, dp, [s], pixels_per_item=ppi)
        for a, b in zip(ref, cel.elbo_grad_hess(one)):
            assert np.array_equal(a[s], b.cpu().numpy()[0])
        for a, b in zip(val, cel.elbo(one)):
            assert np.array_equal(a[s], b.cpu().numpy()[0])
        delta, status = cel.newton_state(dp)
        cel.newton_step(one, delta, status)
        assert int(status[s]) == st[s] and np.array_equal(dp.theta[s].cpu().numpy(), theta[s])
    ctx.synchronize()
