"""The pixel kernels leave out galaxy pairs that are exactly zero at all of a
warp's pixels (beyond the pair's skip radius exp2 underflows to zero)."""
import dataclasses

import numpy as np
import pytest
import torch

import fields
import oracle
from oracle import elbo as OE

f32 = np.float32


def _radius2(P, lw):
    """The kernels' squared skip radius in FP32, from the staged coefficients
    A = -log2(e) / 2 (P11, 2 P12, P22)."""
    h = f32(0.72134752044448170368)
    a, b, d = h * P[..., 0], h * P[..., 1], h * P[..., 2]
    det = a * d - b * b
    lmax = f32(0.5) * (a + d + np.sqrt((a - d) * (a - d) + f32(4) * b * b))
    ok = (a > 0) & (d > 0) & (det > f32(1e-3) * a * d) & (lw < np.inf)
    with np.errstate(all="ignore"):
        return np.where(ok, f32(1.001) * np.maximum(lw + f32(128), 0) * (lmax / det), np.inf)


def test_densities_underflow_beyond_the_radius():
    rng = np.random.default_rng(4)
    n = 20000
    phi = rng.uniform(0, np.pi, n)
    l1 = np.exp(rng.uniform(np.log(0.05), np.log(3e3), n))
    l2 = l1 * np.exp(rng.uniform(np.log(1e-5), 0, n))
    c, s = np.cos(phi), np.sin(phi)
    P = np.stack([c * c / l1 + s * s / l2, c * s * (1 / l1 - 1 / l2), s * s / l1 + c * c / l2], 1).astype(f32)
    lw = np.concatenate([rng.uniform(-60, 10, n - 4), [-200, -np.inf, np.nan, np.inf]]).astype(f32)
    r2 = _radius2(P, lw)
    assert np.isinf(r2[-2:]).all() and (r2[-4:-2] == 0).all()
    fin = np.isfinite(r2) & np.isfinite(lw)
    assert fin.mean() > 0.5                       # elongations up to ~30 have a radius
    for t in rng.uniform(0, np.pi, 64):           # just outside, in FP32 as the kernels evaluate it
        r = np.sqrt(r2[fin] * f32(1.0001))
        dx, dy = (r * np.cos(t)).astype(f32), (r * np.sin(t)).astype(f32)
        h = f32(-0.72134752044448170368)
        p = P[fin]
        arg = lw[fin] + (h * p[:, 0]) * (dx * dx) + (f32(2) * h * p[:, 1]) * (dx * dy) + (h * p[:, 2]) * (dy * dy)
        assert (arg < -126).all()


@pytest.mark.gpu
@pytest.mark.parametrize("n_exp,n_dev,side,psf", [(8, 8, 101, 0.15), (8, 8, 15, 1.0), (3, 8, 61, 0.15),
                                                  (8, 1, 61, 0.3), (5, 6, 33, 0.02)])
def test_far_pixels_match_oracle(n_exp, n_dev, side, psf):
    """Narrow PSFs and a small galaxy: most pairs vanish away from the centre."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1803_00113_gb300 import celeste as cel
    m = fields.make_model()
    m = dataclasses.replace(m, alpha_exp=m.alpha_exp[-n_exp:], tau_exp=m.tau_exp[-n_exp:],
                            alpha_dev=m.alpha_dev[-n_dev:], tau_dev=m.tau_dev[-n_dev:])
    p = fields.plain_source(side=side, bands=1, star=False, model=m)
    p.img_psf[:, :, 3:] *= psf
    p.theta[0, fields.I_LOGRADIUS] = 0.0
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p)
    plan = cel.Plan(ctx, dp, [0])
    e, er, g, H = (t.cpu().numpy()[0] for t in cel.elbo_grad_hess(plan))
    _, er1, g1 = (t.cpu().numpy()[0] for t in cel.elbo_grad(plan))
    er0 = float(cel.elbo(plan)[1])
    E, V = (t.cpu().numpy().astype(np.float64) for t in cel.render(plan))
    ctx.synchronize()
    ref, sc = oracle.elbo_grad_hess(p, 0), oracle.abs_sum_scales(p, 0)
    # tolerances of the parity tests: 1e-5 on values, 1e-4 on derivatives, of
    # the summed magnitudes
    for v in (er, er1, er0):
        assert abs(v - ref["elbo_rel"]) <= 1e-5 * max(abs(ref["elbo_rel"]), sc["elbo"])
    for v in (g, g1):
        assert (np.abs(v - ref["grad"]) <= 1e-4 * np.maximum(np.abs(ref["grad"]), sc["grad"])).all()
    # (type, fluxes and geometry; one band says nothing about the colours,
    # whose entries are the KL's alone)
    k = np.r_[0:5, 21:27]
    ok = np.abs(H - ref["hess"]) <= 1e-4 * np.maximum(np.abs(ref["hess"]), sc["hess"])
    assert ok[np.ix_(k, k)].all()
    (Es, Vs), = OE.render_source_patch(p, 0)
    np.testing.assert_allclose(E, Es.numpy(), rtol=2e-5, atol=1e-6 * float(Es.max()))
    np.testing.assert_allclose(V, Vs.numpy(), rtol=2e-5, atol=1e-6 * float(Vs.max()))
