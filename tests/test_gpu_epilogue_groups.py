"""The per-source epilogue takes pairs in groups of 12 and their tiles in
chunks of 32: sources on either side of both, against the oracle."""
import numpy as np
import pytest
import torch

import fields
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,per_band,side,ppi,pairs", [
    (3, 1, 15, 256, (5, 5)),      # one tile a pair
    (5, 4, 15, 32, (12, 12)),     # a full group; tiles of a pair straddle the chunks
    (6, 4, 15, 64, (13, 20)),     # a second group, partly filled
    (9, 6, 15, 32, (25, 30)),     # three groups
    (4, 1, 41, 32, (5, 5)),       # 53 tiles a pair: several chunks
])
def test_pair_groups_and_tile_chunks(seed, per_band, side, ppi, pairs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    for s in range(seed, seed + 4000):            # the first scene with that many pairs
        p = fields.batched(seed=s, n_sources=1, min_side=side, max_side=side,
                           max_images_per_band=per_band)
        if pairs[0] <= p.n_patches <= pairs[1]:
            break
    assert pairs[0] <= p.n_patches <= pairs[1]
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    plan = cel.Plan(ctx, dp, [0], pixels_per_item=ppi)
    e, er, g, H = (t.cpu().numpy()[0] for t in cel.elbo_grad_hess(plan))
    e1, er1, g1 = (t.cpu().numpy()[0] for t in cel.elbo_grad(plan))
    ctx.synchronize()
    ref, sc = oracle.elbo_grad_hess(p, 0), oracle.abs_sum_scales(p, 0)
    # the parity tests' tolerances: 1e-5 on values, 1e-4 on derivatives
    for v in (e, e1):
        assert abs(v - ref["elbo"]) <= 1e-5 * abs(ref["elbo"])
    for v in (er, er1):
        assert abs(v - ref["elbo_rel"]) <= 1e-5 * max(abs(ref["elbo_rel"]), sc["elbo"])
    for v in (g, g1):
        assert (np.abs(v - ref["grad"]) <= 1e-4 * np.maximum(np.abs(ref["grad"]), sc["grad"])).all()
    assert (np.abs(H - ref["hess"]) <= 1e-4 * np.maximum(np.abs(ref["hess"]), sc["hess"])).all()
