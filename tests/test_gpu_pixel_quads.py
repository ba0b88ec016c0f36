"""The pixel-weight fit with four chains per CTA (many galaxies) against two per CTA (few): the same draws, over the
row-group edges of both layouts' largest sides, mixed sides under one maximum, and chain counts that leave
chain slots empty."""
import numpy as np
import pytest
import torch

import datagen
from paper_2604_22048_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides,chains", [((47, 41, 39, 33), 4), ((31, 25, 17, 7, 3), 4), ((47, 15, 33), 3), ((29, 23), 7)])
def test_four_chains_per_cta(cuda, sides, chains):
    k = len(sides)
    truth = synth.draw_ragged(k, seed=chains)
    truth.side = np.asarray(sides, dtype=np.int64)
    ds = datagen.make_dataset(truth, chains)
    flat, offs, sd = datagen.pack(ds)
    w = np.random.default_rng(k).uniform(0.3, 2.0, flat.shape).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    psf = api.psf_table("moffat", truth.psf_fwhm.astype(np.float32), truth.psf_beta, device=cuda)
    cfg = api.FitConfig(n_chains=chains, n_warmup=20, n_samples=8, n_leapfrog=5, seed=3)
    ids = torch.arange(k, dtype=torch.int64, device=cuda)
    few = api.fit_galaxies(t(flat), t(offs), t(sd), psf, t(ds.sigma.astype(np.float32)), t(ds.init.astype(np.float32)), cfg,
                           gal_id=ids, pixel_weight=t(w), max_side=max(sides))
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    rep = 2 * sms // k                     # two full waves of four-chain CTAs, four of two-chain CTAs
    idx = torch.arange(k, device=cuda).repeat(rep)
    table, n_psf = psf
    table = torch.cat([table.reshape(k, -1)] * rep).reshape((-1,) + tuple(table.shape[1:]))
    many = api.fit_galaxies(t(flat), t(offs)[idx], t(sd)[idx], (table, n_psf * rep),
                            t(ds.sigma.astype(np.float32))[idx], t(ds.init.astype(np.float32))[idx], cfg, gal_id=ids[idx],
                            pixel_weight=t(w), max_side=max(sides))
    for name in ("samples", "logp", "step_size", "inv_mass", "n_grad", "status"):
        a, b = few[name], many[name]
        if name == "samples":
            a, b = a.transpose(0, 1), b.transpose(0, 1)
        assert torch.equal(a[idx], b), name
    assert int(few["status"].max()) == 0
