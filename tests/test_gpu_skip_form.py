"""The derivative kernel's form that leaves out vanished pairs runs for launches of
more than 16 items an SM with patches of 2,048 pixels and more on average.
Its results, source by source: the bits that the source's own plan gives,
which takes the forms without it, and the oracle's values."""
import dataclasses

import numpy as np
import pytest
import torch

import fields
import oracle

pytestmark = pytest.mark.gpu


def _grid(n, side, n_exp, n_dev, psf):
    """n sources of different shapes, side by side, with narrow PSFs."""
    m = fields.make_model()
    m = dataclasses.replace(m, alpha_exp=m.alpha_exp[-n_exp:], tau_exp=m.tau_exp[-n_exp:],
                            alpha_dev=m.alpha_dev[-n_dev:], tau_dev=m.tau_dev[-n_dev:])
    cols = int(np.ceil(np.sqrt(n)))
    p = fields.plain_source(side=cols * side, bands=1, star=False, model=m, sky_grid=(2, 3))
    p.img_psf[:, :, 3:] *= psf
    rng = np.random.default_rng(5)
    k = np.arange(n)
    x0, y0 = (k % cols) * side, (k // cols) * side
    p.theta = np.repeat(p.theta, n, 0)
    # centres anywhere in the middle half: the far corner is up to 3/4 of the patch away
    p.theta[:, fields.I_U] = x0 + side * rng.uniform(0.25, 0.75, n)
    p.theta[:, fields.I_U + 1] = y0 + side * rng.uniform(0.25, 0.75, n)
    p.theta[:, fields.I_LOGRADIUS] = rng.uniform(-0.5, 1.5, n)
    p.theta[:, fields.I_ANGLE] = rng.uniform(0, np.pi, n)
    p.theta[:, fields.I_AXIS] = rng.uniform(-1.5, 1.5, n)
    p.patch_ptr = np.arange(n + 1, dtype=np.int32)
    p.patch_img = np.zeros(n, np.int32)
    p.patch_x0, p.patch_y0 = x0.astype(np.int32), y0.astype(np.int32)
    p.patch_w = p.patch_h = np.full(n, side, np.int32)
    p.nbr_ptr, p.nbr_idx = np.zeros(n + 1, np.int32), np.zeros(0, np.int32)
    return p


@pytest.mark.parametrize("n,side,ppi,n_exp,n_dev,psf,queue", [
    (64, 61, 96, 8, 8, 0.15, False),     # 39 items a patch, the last of 73 pixels
    (64, 101, 256, 8, 8, 0.15, False),   # 40, the last of 217
    (64, 61, 96, 3, 8, 0.3, False),      # five components without a partner
    (64, 61, 96, 8, 1, 0.15, False),     # one pair, seven without
    (40, 46, 32, 5, 6, 0.02, False),     # 67, the last of 4; just above 2,048 pixels
    (110, 61, 32, 8, 8, 0.15, True),     # a pass an item, through the work queue
])
def test_skip_form_equals_the_others(n, side, ppi, n_exp, n_dev, psf, queue):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    items = n * -(-side * side // ppi)
    assert side * side >= 2048 and items > 16 * n_sm, "the launch takes the form with the skip"
    assert queue == (items >= 5 * 4 * 4 * n_sm)
    p = _grid(n, side, n_exp, n_dev, psf)
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    all_ = [t.cpu().numpy() for t in cel.elbo_grad_hess(cel.Plan(ctx, dp, list(range(n)),
                                                                 pixels_per_item=ppi))]
    for s in range(0, n, 3):
        one = cel.elbo_grad_hess(cel.Plan(ctx, dp, [s], pixels_per_item=ppi))
        for a, b in zip(all_, one):
            assert np.array_equal(a[s], b.cpu().numpy()[0])
    ctx.synchronize()
    # the parity tests' tolerances: 1e-5 on values, 1e-4 on derivatives, of the
    # summed magnitudes (one band: type, fluxes and geometry)
    k = np.r_[0:5, 21:27]
    for s in (0, n // 2):
        ref, sc = oracle.elbo_grad_hess(p, s), oracle.abs_sum_scales(p, s)
        assert abs(all_[1][s] - ref["elbo_rel"]) <= 1e-5 * max(abs(ref["elbo_rel"]), sc["elbo"])
        assert (np.abs(all_[2][s] - ref["grad"]) <= 1e-4 * np.maximum(np.abs(ref["grad"]), sc["grad"])).all()
        ok = np.abs(all_[3][s] - ref["hess"]) <= 1e-4 * np.maximum(np.abs(ref["hess"]), sc["hess"])
        assert ok[np.ix_(k, k)].all()
