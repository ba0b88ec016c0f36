"""Shear passes whose log weights span a wide range, at several points and with per-sample offsets: narrow ellipticity
distributions (alpha from 0.005 up, on either side of 0.173, from where no weight can be far above another), samples on and
outside the unit circle (BA14 gives them a weight), galaxies whose first samples have none, and widely scattered offsets
in both families.  Against one point at a time, which rescales as it goes, or the oracle.  Bounds as for the several-point kernel
on ordinary data: 1e-6 of the larger of the point's largest output and one per galaxy; against the oracle 1e-5 and
1e-4 of the gradient's max-norm.  The time of a pass does not depend on the data: 1.6 times the ordinary pass is
allowed (a lane that takes its samples again makes it 2.5)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu
FAMILIES = [O.EPRIOR_BA14, O.EPRIOR_TRUNC_GAUSS]


def _rows(n, K, seed):
    rng = np.random.default_rng(seed)
    e1, e2 = rng.normal(0, 0.15, (2, n, K)).astype(np.float32).clip(-0.45, 0.45)
    e1[::5, :min(K - 1, 9)] = 0.85             # outside the truncation radius: a lane's first samples
    e1[3::10, :min(K - 1, 12)] = 0.85          # a lane's whole first chunk
    return e1, e2


@pytest.mark.parametrize("K", [4, 48, 52, 300])
@pytest.mark.parametrize("family", FAMILIES)
@pytest.mark.parametrize("alphas", [(0.2, 0.3, 0.12, 0.15), (0.107, 0.105, 0.2, 0.02), (0.005, 0.01, 0.05, 0.1),
                                    (0.172, 0.175, 0.2, 0.18)])
def test_points_at_any_width(cuda, K, family, alphas):
    n = 70
    e1, e2 = _rows(n, K, K)
    if family == O.EPRIOR_BA14:
        e1[1::7, K // 2:] = 1.1
        e1[2::7], e2[2::7] = 0.0, 3.5
    t = lambda a: torch.from_numpy(a).to(cuda)
    plan = api.ShearPlan(t(e1), t(e2), family=family, trunc_r=0.7)
    pts = np.column_stack([[0.02, 0.0, -0.03, 0.01], [-0.01, 0.0, 0.02, 0.01], alphas])
    one = np.array([plan.loglike(*p, host=True) for p in pts])
    many = plan.loglike_multi(pts)
    assert np.isfinite(many).all()
    assert (np.abs(many - one).max(1) <= 1e-6 * np.abs(one).max(1).clip(n)).all()
    alone = np.concatenate([plan.loglike_multi(pts[i:i + 1]) for i in range(4)])
    inside = e1.max() < 1.0 and e2.max() < 1.0
    if inside:                                  # a point's result does not depend on the others of its pass
        assert np.array_equal(many, alone)


@pytest.mark.parametrize("family", FAMILIES)
@pytest.mark.parametrize("K", [4, 48, 52, 300, 99])
@pytest.mark.parametrize("spread", [1.0, 100.0])
def test_scattered_offsets(cuda, family, K, spread):
    n = 40
    e1, e2 = _rows(n, K, K + 1)
    b = (spread * np.random.default_rng(K).normal(size=(n, K))).astype(np.float32)
    b[1::4] = np.sort(b[1::4], axis=1)          # weights that rise along the galaxy
    t = lambda a: torch.from_numpy(a).to(cuda)
    plan = api.ShearPlan(t(e1), t(e2), t(b), family=family, trunc_r=0.7)
    for p in ([0.02, -0.01, 0.2], [0.01, 0.02, 0.05]):
        got = plan.loglike(*p, host=True)
        v, g = O.shear_loglike(e1, e2, *p, family=family, b=b)
        assert abs(got[0] - v) <= 1e-5 * max(abs(v), n), (got[0], v)
        assert np.abs(got[1:] - g).max() <= 1e-4 * np.abs(g).max(), (got, g)


def _time(f):
    for _ in range(3):
        f()
    a, b = torch.cuda.Event(True), torch.cuda.Event(True)
    best = 1e9
    for _ in range(5):
        a.record()
        for _ in range(20):
            f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("offsets", [False, True])
def test_time_does_not_depend_on_the_width(cuda, offsets):
    gen = torch.Generator(device=cuda)
    gen.manual_seed(1)
    e1, e2, b = [0.1 * torch.randn((100000, 300), device=cuda, generator=gen) for _ in range(3)]
    plan = api.ShearPlan(e1, e2, b if offsets else None, family=O.EPRIOR_TRUNC_GAUSS, trunc_r=0.7)
    if offsets:
        t = [_time(lambda: plan.loglike(0.02, -0.01, a)) for a in (0.2, 0.02)]
    else:
        pts = [np.column_stack([np.linspace(-0.03, 0.03, 4), np.zeros(4), np.full(4, a)]) for a in (0.2, 0.02)]
        t = [_time(lambda: plan.loglike_multi(p, host=False)) for p in pts]
    assert t[1] <= 1.6 * t[0], t
