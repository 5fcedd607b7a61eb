"""The value epilogue adds an item a thread: three pairs or more of up to 96 items
each are loaded eight pairs together, fewer or longer ones a pair at a time.
Either side of those lines, against the oracle; and a block of it holds less than a
kilobyte of shared memory, not the derivative passes' buffers."""
import os
import subprocess

import numpy as np
import pytest
import torch

import fields
import oracle
from oracle import elbo as OE
from paper_1803_00113_gb300 import build_lib


@pytest.mark.gpu
@pytest.mark.parametrize("bands,side,ppi", [
    (1, 15, 256),     # one pair, one item
    (2, 55, 32),      # two pairs of 95 items
    (3, 15, 256),     # three: loaded together
    (3, 55, 32),      # three of 95 items
    (3, 56, 32),      # three of 98: a pair at a time
    (5, 33, 64),      # five of 18
    (5, 101, 32),     # five of 319
])
def test_value_matches_oracle(bands, side, ppi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = fields.plain_source(side=side, bands=bands, star=False)
    ctx = cel.Context(p.model)
    plan = cel.Plan(ctx, cel.DeviceProblem(p), [0], pixels_per_item=ppi)
    e, er = (float(t[0]) for t in cel.elbo(plan))
    ll = float(cel.loglik(plan)[0])
    _, er2, _, _ = (t.cpu().numpy()[0] for t in cel.elbo_grad_hess(plan))
    ctx.synchronize()
    ref, sc = oracle.elbo_grad_hess(p, 0), oracle.abs_sum_scales(p, 0)
    # the parity tests' tolerance on values: 1e-5 of the summed magnitudes
    tol = 1e-5 * max(abs(ref["elbo_rel"]), sc["elbo"])
    assert abs(e - ref["elbo"]) <= 1e-5 * abs(ref["elbo"])
    assert abs(er - ref["elbo_rel"]) <= tol and abs(er2 - er) <= 2 * tol
    # the pixel part: L_rel without the KL, which depends on theta alone
    assert abs(ll - er - float(OE.kl_source(OE.Theta.from_vector(torch.from_numpy(p.theta[0])), p.model))) <= 2 * tol


@pytest.mark.gpu
@pytest.mark.parametrize("n_images", [7, 8, 9, 17])
def test_groups_of_eight_pairs(n_images):
    """The same patch in n images: the value is n times a patch's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    p = fields.plain_source(side=21, bands=1, star=False)
    ctx = cel.Context(p.model)
    one = float(cel.loglik(cel.Plan(ctx, cel.DeviceProblem(p), [0]))[0])
    p.patch_ptr = np.array([0, n_images], np.int32)
    for k in ("patch_img", "patch_x0", "patch_y0", "patch_w", "patch_h"):
        setattr(p, k, np.repeat(getattr(p, k), n_images))
    many = float(cel.loglik(cel.Plan(ctx, cel.DeviceProblem(p), [0]))[0])
    ctx.synchronize()
    assert abs(many - n_images * one) <= 1e-12 * abs(many)    # FP64 sums of equal terms


def test_block_of_the_value_epilogue_is_small(tmp_path):
    nvcc = build_lib._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "size.cu"
    src.write_text('#include "epilogue.cuh"\nusing namespace celeste;\n'
                   'static_assert(sizeof(EpiShared<0>) <= 1024, "");\n')
    r = subprocess.run([nvcc, *build_lib.ARCH, "-std=c++17", f"-I{build_lib.INCLUDE}",
                        f"-I{build_lib.CSRC}", "-c", str(src), "-o", str(tmp_path / "size.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
