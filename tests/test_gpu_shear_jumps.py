"""Log weights that jump by more than 2^32 inside a galaxy, and galaxies whose first samples all have zero weight, at several
points per pass: the tile kernel sums against the first four samples' reference and takes such a lane's samples again at the
galaxy's end; the same points one at a time go through the kernel that rescales as it goes (itself held to the oracle on
such data by the parity tests).  Bound: 1e-6 of the larger of the point's largest output and one per galaxy, as for
the several-point kernel on ordinary data.  K = 99 takes the register kernels."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu

POINTS = np.array([[0.02, -0.01, 0.2], [0.0, 0.0, 0.03], [-0.03, 0.02, 0.025], [0.01, 0.01, 0.3], [0.0, 0.02, 0.04]])


@pytest.mark.parametrize("K", [4, 48, 52, 100, 300, 99])
@pytest.mark.parametrize("family", [O.EPRIOR_BA14, O.EPRIOR_TRUNC_GAUSS])
def test_jumps_at_several_points(cuda, K, family):
    rng = np.random.default_rng(K)
    n = 70
    e1, e2 = rng.normal(0, 0.2, (2, n, K)).astype(np.float32).clip(-0.45, 0.45)
    e1[::3, :min(K - 1, 20)] = 0.8          # beyond the truncation radius: zero weight
    e2[::3, :min(K - 1, 20)] = 0.1
    order = np.argsort(-np.hypot(e1[1::3], e2[1::3]), axis=1)   # weights that rise along the galaxy
    e1[1::3] = np.take_along_axis(e1[1::3], order, 1)
    e2[1::3] = np.take_along_axis(e2[1::3], order, 1)
    t = lambda a: torch.from_numpy(a).to(cuda)
    plan = api.ShearPlan(t(e1), t(e2), family=family, trunc_r=0.7)
    one = np.array([plan.loglike(*p, host=True) for p in POINTS])
    many = plan.loglike_multi(POINTS)
    assert np.isfinite(many).all()
    assert (np.abs(many - one).max(1) <= 1e-6 * np.abs(one).max(1).clip(n)).all()
