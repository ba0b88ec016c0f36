"""Chain diagnostics of samples in any unit: the ESS and R-hat do not depend on the scale, down to variances below the
smallest normal float.  At 2^-66 the products of deviations are denormal, spaced 2^-17 of their size: a lag's rho is off by
about 2^-16, and a sum of ten of them moves tau, and with it the ESS, by 1e-3 at most; 1e-2 allowed."""
import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import api
from test_gpu_ess_sizes import _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-66, -64, -40, 40, 58])
def test_ess_of_small_and_large_units(cuda, exponent):
    rng = np.random.default_rng(4)
    n, C, S = 2, 4, 300
    phi = np.array([-0.3, 0.0, 0.3, 0.5, 0.7, 0.8])[:, None, None]
    x = rng.normal(size=(6, n, C, S))
    for t in range(1, S):
        x[..., t] = phi * x[..., t - 1] + np.sqrt(1 - phi ** 2) * x[..., t]
    x = (x.astype(np.float32) * np.float32(2.0 ** exponent)).astype(np.float32)
    ess, rh = [a.cpu().numpy() for a in api.chain_ess(torch.from_numpy(x).to(cuda))]
    for k in range(6):
        for g in range(n):
            e, r = _reference(x[k, g].astype(np.float64) * 2.0 ** -exponent)
            assert abs(ess[g, k] - e) <= 1e-2 * e, (k, g, ess[g, k], e)
            assert abs(rh[g, k] - r) <= 1e-3 * r


@pytest.mark.parametrize("S", [28664, 28665, 28668])
def test_one_chain_on_either_side_of_shared_memory(cuda, S):
    """One chain takes the room of two: 2 (S + 8) floats of 224 KB.  Bounds as for the other lengths (the sums of the
    ESS in float32: 2e-4 relative)."""
    rng = np.random.default_rng(S)
    x = (2.0 + 0.1 * rng.normal(size=(6, 1, 1, S))).astype(np.float32)
    ess, rh = [a.cpu().numpy() for a in api.chain_ess(torch.from_numpy(x).to(cuda))]
    for k in range(6):
        e, r = _reference(x[k, 0])
        assert abs(ess[0, k] - e) <= 2e-4 * e and abs(rh[0, k] - r) <= 1e-5 * r
