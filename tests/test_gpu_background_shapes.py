"""Backgrounds over overlaps narrower than a chunk's rows (patches wider than a
chunk, chunks inside a row or across two), with items shared by two or four
warps or by none, and of plans without neighbours (the sky alone): the same
bits as the gather from a render cache."""
import numpy as np
import pytest
import torch

import fields

pytestmark = pytest.mark.gpu


def _scene(n, w, h, sx, sy):
    """n sources with w x h patches, (sx, sy) pixels apart, in one band's image."""
    p = fields.plain_source(side=max(w + sx * n, h + sy * n, 64), bands=1, star=False, sky_grid=(2, 3))
    k = np.arange(n)
    p.theta = np.repeat(p.theta, n, 0)
    p.theta[:, fields.I_U] = sx * k + w / 2
    p.theta[:, fields.I_U + 1] = sy * k + h / 2
    p.patch_ptr = np.arange(n + 1, dtype=np.int32)
    p.patch_img = np.zeros(n, np.int32)
    p.patch_x0, p.patch_y0 = (sx * k).astype(np.int32), (sy * k).astype(np.int32)
    p.patch_w, p.patch_h = np.full(n, w, np.int32), np.full(n, h, np.int32)
    nb = [[t for t in range(n) if t != s and abs(t - s) * sx < w and abs(t - s) * sy < h] for s in range(n)]
    p.nbr_ptr = np.concatenate([[0], np.cumsum([len(b) for b in nb])]).astype(np.int32)
    p.nbr_idx = np.array([t for b in nb for t in b], np.int32)
    return p


@pytest.mark.parametrize("n,w,h,sx,sy,ppi", [
    (2, 300, 5, 200, 0, 256),      # chunks in a row and across two
    (2, 1000, 3, 700, 1, 256),     # a quarter of a row a chunk
    (2, 1000, 3, 700, 1, 1024),
    (3, 257, 4, 200, 1, 128),
    (2, 256, 4, 190, 0, 256),      # exactly a row
    (2, 255, 4, 190, 1, 64),
    (2, 33, 65, 0, 48, 32),        # items of less than a row
    (2, 33, 65, 0, 48, 100),
    (9, 101, 40, 80, 0, 256),      # overlaps of a fifth of a row
    (60, 90, 70, 70, 0, 64),       # more items than are shared
    (1, 1, 1, 0, 0, 256),          # no neighbours from here on
    (1, 31, 33, 0, 0, 32),
    (3, 31, 33, 31, 0, 256),
    (1, 333, 7, 0, 0, 1024),
    (150, 40, 40, 40, 0, 64),      # 3,750 items
])
def test_background_equals_the_gather(n, w, h, sx, sy, ppi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = _scene(n, w, h, sx, sy)
    ctx = cel.Context(p.model)
    got = []
    for cached in (False, True):
        dp = cel.DeviceProblem(p, render_cache=cached)
        plan = cel.Plan(ctx, dp, list(range(n)), pixels_per_item=ppi)
        if cached:
            cel.render_cache(plan)
        got.append([t.cpu().numpy() for t in cel.background(plan)])
    ctx.synchronize()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_sky_alone_reports_a_sky_of_zero():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = _scene(1, 20, 20, 0, 0)
    p.sky = np.zeros_like(p.sky)
    ctx = cel.Context(p.model)
    cel.background(cel.Plan(ctx, cel.DeviceProblem(p), [0]))
    with pytest.raises(cel.CelesteError):
        ctx.synchronize()
