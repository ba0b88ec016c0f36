"""Chain diagnostics where the kernel's layout changes: odd and even chain counts, lengths around the lanes' runs and the
lag blocks, 16-byte loads and not, chains too long for shared memory; against a float64 numpy version.  The sums over a
chain are in float32: 2e-4 relative on the ESS (tau is near the difference of two such sums), 1e-5 on R-hat."""
import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu


def _reference(x):
    C, S = x.shape
    x = x.astype(np.float64)
    d = x - x.mean(1, keepdims=True)
    W = (d ** 2).sum(1).mean() / (S - 1)
    vp = (S - 1) / S * W + (x.mean(1).var(ddof=1) if C > 1 else 0.0)
    rho = lambda t: 1.0 - (W - sum((d[c, :S - t] * d[c, t:]).sum() / S for c in range(C)) / C) / vp
    total, prev, k = 0.0, np.inf, 0
    while 2 * k + 1 < S:
        P = (1.0 if k == 0 else rho(2 * k)) + rho(2 * k + 1)
        if not P > 0:
            break
        prev = min(prev, P)
        total += prev
        k += 1
    tau = max(-1.0 + 2.0 * total, 1.0 / np.log10(C * S))
    return C * S / tau, np.sqrt(vp / W)


@pytest.mark.parametrize("C,S", [(1, 4), (1, 5), (2, 9), (3, 31), (4, 32), (5, 33), (8, 64), (3, 97), (4, 300), (8, 600),
                                 (7, 1201), (2, 20000), (8, 7160), (8, 7200)])
def test_ess_over_layouts(cuda, C, S):
    rng = np.random.default_rng(100 * C + S)
    n = 3
    phi = np.array([-0.4, 0.0, 0.3, 0.7, 0.9, 0.97])[:, None, None]
    x = rng.normal(size=(6, n, C, S))
    for t in range(1, S):
        x[..., t] = phi * x[..., t - 1] + np.sqrt(1 - phi ** 2) * x[..., t]
    x = (2.8 + 0.05 * x).astype(np.float32)
    ess, rh = [a.cpu().numpy() for a in api.chain_ess(torch.from_numpy(x).to(cuda))]
    for k in range(6):
        for g in range(n):
            e, r = _reference(x[k, g])
            assert abs(ess[g, k] - e) <= 2e-4 * e, (k, g, ess[g, k], e)
            assert abs(rh[g, k] - r) <= 1e-5 * r


def test_constant_chains(cuda):
    ess, rh = api.chain_ess(torch.ones((6, 2, 3, 50), device=cuda))
    assert torch.isnan(rh).all() and torch.isfinite(ess).all()
