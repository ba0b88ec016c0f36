"""The per-pixel-weight evaluation over every number of eight-row groups its products and epilogues take (1 to 8 over the side,
1 to 4 over the half plane), smaller stamps in a launch of a larger maximum, and odd chain counts; against the oracle's
pixel-space likelihood (1e-5 relative on the log posterior, 1e-4 of the gradient's max-norm, as in the parity tests)."""
import numpy as np
import pytest
import torch

import datagen
import oracle as O
from paper_2604_22048_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", [[3, 7, 9, 15, 17, 23, 25, 31], [33, 39, 41, 47, 49, 55, 57, 63], [5, 63, 31, 33]])
def test_logpost_over_row_groups(cuda, sides):
    truth = synth.draw_ragged(len(sides), seed=len(sides))
    truth.side = np.asarray(sides, dtype=np.int64)
    ds = datagen.make_dataset(truth, 3)
    flat, offs, sd = datagen.pack(ds)
    rng = np.random.default_rng(sides[0])
    w = rng.uniform(0.3, 2.0, flat.shape).astype(np.float32)
    w[rng.random(flat.shape) < 0.02] = 0.0
    pts = (ds.theta + rng.normal(0, [0.02, 0.02, 0.03, 0.03, 0.05, 0.05], ds.theta.shape)).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    psf = api.psf_table("moffat", truth.psf_fwhm.astype(np.float32), truth.psf_beta, device=cuda)
    args = (t(flat), t(offs), t(sd), psf, t(ds.sigma.astype(np.float32)))
    lp, g = [x.cpu().numpy() for x in api.logpost_points(*args, t(np.arange(len(sides), dtype=np.int32)), t(pts),
                                                         pixel_weight=t(w))]
    for i, N in enumerate(sides):
        d = flat[offs[i]:offs[i] + N * N].astype(np.float64).reshape(N, N)
        wi = w[offs[i]:offs[i] + N * N].astype(np.float64).reshape(N, N)
        ref, gref = O.logpost(N, 0.2, ds.psf[i], d, 1.0, pts[i].astype(np.float64), weights=wi)
        assert abs(lp[i] - ref) <= 1e-5 * abs(ref), (N, lp[i], ref)
        assert np.abs(g[i] - gref).max() <= 1e-4 * np.abs(gref).max() + 1e-3, (N, g[i], gref)
    cfg = api.FitConfig(n_chains=3, n_warmup=20, n_samples=10, n_leapfrog=5, seed=2)
    r = api.fit_galaxies(*args, t(ds.init.astype(np.float32)), cfg, pixel_weight=t(w))
    assert (r["status"].cpu().numpy() == 0).all()
    last = r["samples"][:, :, :, -1].permute(1, 2, 0).reshape(-1, 6).contiguous()
    gi = torch.arange(len(sides), dtype=torch.int32, device=cuda).repeat_interleave(3)
    again, _ = api.logpost_points(*args, gi, last, pixel_weight=t(w))
    stored = r["logp"][:, :, -1].reshape(-1).double()
    # the stored value belongs to the compensated position, the sample is its float
    assert (torch.abs(stored - again) <= 1e-5 * again.abs()).all()
