"""Neighbour backgrounds go over the overlap of each neighbour's patch with a
chunk of 256 pixels (rendered) or through asynchronous copies from the render
cache: sizes on either side of the chunk, overlaps of one pixel and one row,
more neighbours than copies in flight and than lanes, against the oracle and
against each other."""
import numpy as np
import pytest
import torch

import fields
from oracle import elbo as OE

pytestmark = pytest.mark.gpu


def _scene(n, side, step, ppi_w=64):
    """n sources on a diagonal, step pixels apart, in one band's image."""
    p = fields.plain_source(side=max(side + step * n + 8, ppi_w), bands=1, star=False, sky_grid=(2, 3))
    rep = np.repeat
    p.theta = rep(p.theta, n, 0)
    p.theta[:, fields.I_U:fields.I_U + 2] += step * (np.arange(n) - n / 2)[:, None]
    p.patch_ptr = np.arange(n + 1, dtype=np.int32)
    p.patch_img = np.zeros(n, np.int32)
    p.patch_x0 = (step * np.arange(n)).astype(np.int32)
    p.patch_y0 = (step * np.arange(n)).astype(np.int32)
    p.patch_w, p.patch_h = np.full(n, side, np.int32), np.full(n, side, np.int32)
    nb = [[t for t in range(n) if t != s and abs(t - s) * step < side] for s in range(n)]
    p.nbr_ptr = np.concatenate([[0], np.cumsum([len(b) for b in nb])]).astype(np.int32)
    p.nbr_idx = np.array([t for b in nb for t in b], np.int32)
    return p


@pytest.mark.parametrize("n,side,step,ppi", [
    (2, 15, 14, 256),     # one pixel shared, one item
    (3, 16, 5, 256),      # exactly one chunk
    (3, 17, 5, 256),      # a chunk and 33 pixels
    (4, 33, 11, 1024),    # several chunks an item
    (2, 33, 9, 32),       # items of one row and less
    (40, 21, 0, 256),     # 39 neighbours on the same patch
])
def test_backgrounds_match_oracle_and_cache(n, side, step, ppi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = _scene(n, side, step)
    ctx = cel.Context(p.model)
    got = []
    for cached in (False, True):
        dp = cel.DeviceProblem(p, render_cache=cached)
        plan = cel.Plan(ctx, dp, list(range(n)), pixels_per_item=ppi)
        if cached:
            cel.render_cache(plan)
        got.append([t.cpu().numpy() for t in cel.background(plan)])
        E, V = (t.cpu().numpy().astype(np.float64) for t in cel.render(plan))
    ctx.synchronize()
    assert all(np.array_equal(a, b) for a, b in zip(*got))      # the same values, in the same order
    bE, bV = (t.astype(np.float64) for t in got[0])
    for s in (0, n // 2, n - 1):
        (pd,) = OE.gather_patches(p, s)
        (rE, rV), = OE.render_source_patch(p, s)
        sl = slice(s * side * side, (s + 1) * side * side)
        np.testing.assert_allclose(E[sl], rE.numpy(), rtol=2e-5, atol=1e-6 * float(rE.max()))
        np.testing.assert_allclose(V[sl], rV.numpy(), rtol=2e-5, atol=1e-6 * float(rV.max()))
        rbE, rbV = OE.background_patch(p, s, pd)
        np.testing.assert_allclose(bE[sl], rbE.numpy(), rtol=4e-6)
        np.testing.assert_allclose(bV[sl], rbV.numpy(), rtol=2e-5, atol=1e-6 * max(float(rbV.max()), 1.0))
