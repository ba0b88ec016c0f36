"""The dense-covariance fit's chain slots: every chain count, small and the largest stamps, chains that end at
different times, and points in runs that fill the slots or not.  Stored log posteriors against the oracle's Cholesky
solve (1e-5 relative, as in the other parity tests); a point's value does not depend on its run."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_22048_gb300 import api, synth
from test_gpu_dense_cov import PSF, _dataset, _upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chains,sides", [(1, [5, 31]), (2, [9, 17]), (3, [31, 5]), (4, [21, 31])])
def test_fit_every_chain_count(cuda, chains, sides):
    th, covs, stamps = _dataset(sides, 20 + chains)
    data, offs, side, cov, coffs = _upload(sides, covs, stamps, cuda)
    prec, status = api.dense_precision(cov, coffs, side)
    assert (status.cpu().numpy() == 0).all()
    init = torch.from_numpy(np.repeat(np.array(th, np.float32)[:, None], chains, axis=1)).to(cuda).contiguous()
    cfg = api.FitConfig(n_chains=chains, n_warmup=30, n_samples=20, n_leapfrog=6, seed=chains)
    r = api.fit_galaxies(data, offs, side, api.psf_table("moffat", 0.8, 3.0, device=cuda),
                         torch.ones(len(sides), device=cuda), init, cfg, pixel_prec=prec, prec_offsets=coffs)
    samples, logp = r["samples"].cpu().numpy(), r["logp"].cpu().numpy()
    assert (r["status"].cpu().numpy() == 0).all() and np.isfinite(samples).all()
    for i, N in enumerate(sides):
        for ch in range(chains):
            q = samples[:, i, ch, -1].astype(np.float64)
            v, _ = O.loglike_dense(N, 0.2, PSF, stamps[i].astype(np.float64),
                                   covs[i].astype(np.float32).astype(np.float64), q)
            ref = v + O.log_prior(q)
            assert abs(logp[i, ch, -1] - ref) <= 1e-5 * max(abs(ref), 1.0), (N, ch, logp[i, ch, -1], ref)


def test_points_do_not_depend_on_their_run(cuda):
    sides = [13, 5, 31]
    th, covs, stamps = _dataset(sides, 5)
    data, offs, side, cov, coffs = _upload(sides, covs, stamps, cuda)
    prec, _ = api.dense_precision(cov, coffs, side)
    gi = np.repeat([0, 2, 1, 0], [5, 3, 1, 2]).astype(np.int32)
    rng = np.random.default_rng(2)
    pts = (np.array(th)[gi] + rng.normal(0, 0.02, (len(gi), 6))).astype(np.float32)
    pts[1, 2] = 1.5                       # off the prior's support
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    args = (data, offs, side, api.psf_table("moffat", 0.8, 3.0, device=cuda), torch.ones(3, device=cuda))
    kw = dict(pixel_prec=prec, prec_offsets=coffs, max_side=31)
    lp, g = [x.cpu().numpy() for x in api.logpost_points(*args, t(gi), t(pts), **kw)]
    assert np.isneginf(lp[1]) and np.isnan(g[1]).all()
    for i in range(len(gi)):
        one, gone = [x.cpu().numpy() for x in api.logpost_points(*args, t(gi[i:i + 1]), t(pts[i:i + 1]), **kw)]
        assert np.array_equal(lp[i:i + 1], one) and np.array_equal(g[i:i + 1], gone, equal_nan=True)
