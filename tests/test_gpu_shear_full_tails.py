"""The all-free likelihood where its normal-CDF terms change form: samples on either side of mu_f in one galaxy, arguments
around 6 and 14.5 and deep in the left tail, galaxy counts that fill a warp's four or not, sample counts around the blocks of
32; against the oracle (1e-5 of the value, 1e-4 of the gradient's max-norm, as the parity tests)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,a_f", [(1, 1, 14.0), (3, 31, 14.0), (4, 32, -14.0), (5, 33, 14.0), (9, 100, 40.0),
                                     (31, 65, 0.0), (130, 7, 2.0)])
def test_full_matches_oracle(cuda, n, K, a_f):
    rng = np.random.default_rng(n + K)
    e1, e2 = rng.normal(0, 0.15, (2, n, K)).astype(np.float32)
    centre = np.resize([2.45, 2.45 + 0.4 * 6 / 14, 2.45 + 0.4 * 14.5 / 14, 1.2, 3.5], n)[:, None]
    lf = (centre + 0.05 * rng.normal(size=(n, K))).astype(np.float32)
    ls = (-0.4 + 0.05 * rng.normal(size=(n, K))).astype(np.float32)
    th = [0.02, -0.01, 0.22, 2.45, 0.4, a_f, -0.4, 0.06]
    t = lambda a: torch.from_numpy(a).to(cuda)
    for family in (O.EPRIOR_BA14, O.EPRIOR_TRUNC_GAUSS):
        plan = api.ShearPlan(t(e1), t(e2), family=family, trunc_r=0.7)
        v, g = plan.loglike_full(t(lf), t(ls), th)
        rv, rg = O.shear_loglike_full(e1, e2, lf, ls, th, family=family)
        assert abs(v - rv) <= 1e-5 * abs(rv), (v, rv)
        assert np.abs(g - rg).max() <= 1e-4 * np.abs(rg).max(), (g, rg)
