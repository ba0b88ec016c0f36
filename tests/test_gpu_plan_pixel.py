"""An autotuned launch plan with per-pixel weights runs every chain: chain counts that take one, two and four CTAs of two
chains, stamps on either side of the largest of the four-chain layout (47 px); the same draws as the untuned plan's."""
import numpy as np
import pytest
import torch

import datagen
from paper_2604_22048_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chains", [1, 2, 3, 4, 7])
def test_autotuned_plan_runs_every_chain(cuda, chains):
    truth = synth.draw_ragged(4, seed=chains)
    truth.side = np.array([25, 41, 63, 53], dtype=np.int64)
    ds = datagen.make_dataset(truth, chains)
    flat, offs, sd = datagen.pack(ds)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    psf = api.psf_table("moffat", truth.psf_fwhm.astype(np.float32), truth.psf_beta, device=cuda)
    cfg = api.FitConfig(n_chains=chains, n_warmup=20, n_samples=8, n_leapfrog=5, seed=3)
    args = (t(flat), t(offs), t(sd), psf, t(ds.sigma.astype(np.float32)), t(ds.init.astype(np.float32)), cfg)
    kw = dict(pixel_weight=t(np.random.default_rng(1).uniform(0.3, 2.0, flat.shape).astype(np.float32)))
    ref = api.RaggedFitPlan(*args, **kw).run().result()
    plan = api.RaggedFitPlan(*args, autotune=True, **kw)
    out = plan.result()
    names = ("samples", "logp", "step_size", "inv_mass", "n_grad")
    for name in names:
        out[name].fill_(-1)                # what the autotuner's own launches have written
    plan.run()
    torch.cuda.synchronize()
    assert int(out["status"].abs().max()) == 0
    for name in names:
        assert torch.equal(out[name], ref[name]), name


@pytest.mark.parametrize("chains,autotune", [(4, False), (4, True), (3, True)])
def test_plan_with_four_chains_per_cta(cuda, chains, autotune):
    """Enough galaxies that CTAs of four chains take fewer waves: the draws of the few fitted alone."""
    sides = [41, 33, 47]
    k = len(sides)
    truth = synth.draw_ragged(k, seed=10 + chains)
    truth.side = np.array(sides, dtype=np.int64)
    ds = datagen.make_dataset(truth, chains)
    flat, offs, sd = datagen.pack(ds)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    psf = api.psf_table("moffat", 0.8, 3.0, device=cuda)
    w = t(np.random.default_rng(2).uniform(0.3, 2.0, flat.shape).astype(np.float32))
    cfg = api.FitConfig(n_chains=chains, n_warmup=10, n_samples=6, n_leapfrog=5, seed=3)
    ids = torch.arange(k, dtype=torch.int64, device=cuda)
    few = api.fit_galaxies(t(flat), t(offs), t(sd), psf, t(ds.sigma.astype(np.float32)), t(ds.init.astype(np.float32)), cfg,
                           gal_id=ids, pixel_weight=w)
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    idx = torch.arange(2 * sms, device=cuda) % k
    plan = api.RaggedFitPlan(t(flat), t(offs)[idx], t(sd)[idx], psf, t(ds.sigma.astype(np.float32))[idx],
                             t(ds.init.astype(np.float32))[idx], cfg, gal_id=ids[idx], pixel_weight=w, autotune=autotune)
    assert [i["chains_per_cta"] for i in plan.info()] == [4]
    many = plan.run().result()
    for name in ("samples", "logp", "step_size", "inv_mass", "n_grad", "status"):
        a, b = few[name], many[name]
        if name == "samples":
            a, b = a.transpose(0, 1), b.transpose(0, 1)
        assert torch.equal(a[idx], b), name
