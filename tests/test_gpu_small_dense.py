"""Dense-covariance fits and points of small stamps in large numbers: warps per CTA by load and side, several CTAs per SM, the
chains of a galaxy in one CTA or split; the same bits as a few galaxies give in the largest layout, in every one of
them, and a time that follows the stamp (limits between what 16 warps per CTA took and what the present layouts do)."""
import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import api
from test_gpu_dense_cov import _dataset, _upload

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


class _Dense:
    """Four galaxies of one side, repeated to any number; every repetition has its galaxy's random stream."""

    def __init__(self, cuda, side):
        self.cuda, self.n = cuda, 4
        th, covs, stamps = _dataset([side] * self.n, side)
        data, offs, sd, cov, coffs = _upload([side] * self.n, covs, stamps, cuda)
        prec, status = api.dense_precision(cov, coffs, sd)
        assert int(status.abs().max()) == 0
        self.th = torch.from_numpy(np.array(th, np.float32)).to(cuda)
        self.arrays, self.prec, self.side = (data, offs, sd, coffs), prec, side
        self.psf = api.psf_table("moffat", 0.8, 3.0, device=cuda)

    def idx(self, n):
        return torch.arange(n, device=self.cuda) % self.n

    def fit(self, n, chains):
        i = self.idx(n)
        data, offs, sd, coffs = self.arrays
        cfg = api.FitConfig(n_chains=chains, n_warmup=10, n_samples=6, n_leapfrog=5, seed=7)
        return api.FitPlan(data, offs[i], sd[i], self.psf, torch.ones(n, device=self.cuda),
                           self.th[i][:, None].repeat(1, chains, 1).contiguous(), cfg, gal_id=i.contiguous(), max_side=self.side,
                           pixel_prec=self.prec, prec_offsets=coffs[i].contiguous())

    def points(self, gi, th):
        data, offs, sd, coffs = self.arrays
        return api.logpost_points(data, offs, sd, self.psf, torch.ones(self.n, device=self.cuda), gi, th, max_side=self.side,
                                  pixel_prec=self.prec, prec_offsets=coffs)


@pytest.mark.parametrize("side,chains", [(5, 1), (7, 2), (9, 3), (13, 1), (13, 4), (15, 1), (15, 2), (17, 3)])
def test_dense_fit_in_every_layout(cuda, side, chains):
    d = _Dense(cuda, side)
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    ref = d.fit(d.n, chains).run().result()          # a CTA per chain
    assert int(ref["status"].abs().max()) == 0
    # two CTAs per SM, some, and as many as there can be
    for n in (sms - 1, sms + 5, 3 * sms, 9 * sms + 2):
        out = d.fit(n, chains).run().result()
        i = d.idx(n)
        for name in ("samples", "logp", "step_size", "inv_mass", "n_grad", "status"):
            a, b = ref[name], out[name]
            if name == "samples":
                a, b = a.transpose(0, 1), b.transpose(0, 1)
            assert torch.equal(a[i], b), (name, n)


@pytest.mark.parametrize("side", [5, 9, 13, 15, 17])
def test_dense_points_in_every_layout(cuda, side):
    d = _Dense(cuda, side)
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    gen = torch.Generator(device=cuda)
    gen.manual_seed(side)
    few = torch.tensor([0, 1, 1, 2, 2, 2, 3, 3, 3, 3, 0], device=cuda)     # runs of every length
    th = d.th[few] + 0.02 * torch.randn((len(few), 6), device=cuda, generator=gen)
    th[4, 2] = 1.5                                  # off the prior's support
    lp, g = d.points(few.int(), th)
    rep = 5 * sms // len(few) + 1
    lp2, g2 = d.points(few.int().repeat(rep), th.repeat(rep, 1))
    assert torch.equal(lp.repeat(rep), lp2)
    assert torch.equal(g.repeat(rep, 1).nan_to_num(nan=7.0), g2.nan_to_num(nan=7.0))


def test_time_of_many_small_dense_galaxies(cuda):
    d = _Dense(cuda, 7)
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    t = [_time(d.fit(n, 1).run) for n in (sms, 13 * sms)]
    assert t[1] <= 5 * t[0], t
    gi = [torch.arange(n, device=cuda).int() % d.n for n in (sms, 13 * sms)]
    t = [_time(lambda: [d.points(i, d.th[i.long()]) for _ in range(20)]) for i in gi]
    assert t[1] <= 3.5 * t[0], t
