"""Points of galaxies with several exposures or a noise correlation, whose staging keeps one, two or four warps of a CTA busy:
the same bits whatever run of points they come in, on either side of the sides where the number changes, and
a time that follows the staging (a limit between what four idle warps took and what one takes)."""
import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu


def _time(f):
    for _ in range(2):
        f()
    a, b = torch.cuda.Event(True), torch.cuda.Event(True)
    best = 1e9
    for _ in range(5):
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def _folded(cuda, n, side, exposures, corr):
    gen = torch.Generator(device=cuda)
    gen.manual_seed(side)
    size = exposures * side * side
    data = torch.randn(n * size, device=cuda, generator=gen)
    c = None
    if corr:
        c = torch.zeros((n * exposures, side, side), device=cuda)
        m = (side - 1) // 2
        c[:, m, m] = 1.0
        c[:, m, m - 1] = c[:, m, m + 1] = 0.2
        c = c.reshape(-1)
    th = torch.tensor([1.5, -0.3, 0.1, -0.05, 0.1, 0.2], device=cuda) + 0.02 * torch.randn((n, 6), device=cuda, generator=gen)
    return dict(data=data, offsets=torch.arange(n, device=cuda) * size,
                side=torch.full((n,), side, dtype=torch.int32, device=cuda),
                psf=api.psf_table("gaussian", np.array([0.7], np.float32), device=cuda),
                noise_sigma=torch.ones(n * exposures, device=cuda), n_exposures=exposures, noise_corr=c, max_side=side), th


@pytest.mark.parametrize("side,exposures,corr", [(15, 2, True), (31, 3, False), (33, 1, True), (47, 2, False), (49, 2, True)])
def test_folded_points_do_not_depend_on_their_run(cuda, side, exposures, corr):
    kw, th = _folded(cuda, 3, side, exposures, corr)
    gi = torch.tensor([0, 0, 0, 0, 0, 1, 2, 2, 2, 0, 0], device=cuda)
    pts = th[gi] + 0.01 * torch.arange(len(gi), device=cuda)[:, None]
    pts[3, 2] = 1.5
    lp, g = api.logpost_points(gal_index=gi.int(), theta=pts, **kw)
    assert bool(torch.isneginf(lp[3])) and bool(torch.isnan(g[3]).all())
    for i in range(len(gi)):
        one, gone = api.logpost_points(gal_index=gi[i:i + 1].int(), theta=pts[i:i + 1], **kw)
        assert torch.equal(lp[i:i + 1], one) and torch.equal(g[i:i + 1].nan_to_num(nan=7.0), gone.nan_to_num(nan=7.0))


@pytest.mark.parametrize("side,exposures,corr", [(15, 2, True), (25, 3, False)])
def test_time_of_folded_points(cuda, side, exposures, corr):
    """The staging dominates a point as it does a fit of one step, which stages each galaxy with one warp."""
    n = 4000
    kw, th = _folded(cuda, n, side, exposures, corr)
    gi = torch.arange(n, dtype=torch.int32, device=cuda)
    lib_kw = {k: kw[k] for k in ("n_exposures", "noise_corr", "max_side")}
    plan = api.FitPlan(kw["data"], kw["offsets"], kw["side"], kw["psf"], kw["noise_sigma"], th[:, None].contiguous(),
                       api.FitConfig(n_chains=1, n_warmup=0, n_samples=1, n_leapfrog=1), **lib_kw)
    fit = _time(lambda: [plan.run() for _ in range(5)])
    pts = _time(lambda: [api.logpost_points(gal_index=gi, theta=th, **kw) for _ in range(5)])
    assert pts <= 1.2 * fit, (pts, fit)
