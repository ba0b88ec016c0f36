"""The dense precision in batches: one CTA per galaxy and several, clusters that take one galaxy after another (on the scratch
that the last one left, also after one that is not positive definite or whose side is not allowed); the same bits and
status as for a few galaxies, which the other tests hold to numpy's inverse."""
import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import api
from test_gpu_dense_cov import _dataset

pytestmark = pytest.mark.gpu


def _repeat(cuda, covs, sides, idx):
    size = [N ** 4 for N in sides]
    start = np.concatenate([[0], np.cumsum([size[i] for i in idx])[:-1]])
    cov = torch.cat([covs[i] for i in idx])
    side = torch.tensor([sides[i] for i in idx], dtype=torch.int32, device=cuda)
    prec, status = api.dense_precision(cov, torch.from_numpy(start.astype(np.int64)).to(cuda), side, max(N for N in sides if N % 2))
    return [prec[s:s + size[i]] for s, i in zip(start.tolist(), idx)], status.tolist()


@pytest.mark.parametrize("sides,bad", [((5, 7, 9, 11, 13), 1), ((13, 9, 3 + 1, 13, 11), 3), ((17, 5, 15), 2), ((7, 7, 7), 0)])
def test_batches_have_the_bits_of_single_galaxies(cuda, sides, bad):
    """Side 4 stands for one that is refused."""
    odd = [N if N % 2 else N + 1 for N in sides]
    _, covs, _ = _dataset(odd, sum(sides))
    covs[bad][-1, -1] = -1.0                           # the last pivot fails
    covs = [torch.from_numpy(S.astype(np.float32).ravel()[:N ** 4].copy()).to(cuda) for S, N in zip(covs, sides)]
    one = [_repeat(cuda, covs, sides, [i]) for i in range(len(sides)) if sides[i] % 2]
    want, status = {}, {}
    for i, (p, s) in zip([i for i in range(len(sides)) if sides[i] % 2], one):
        want[i], status[i] = p[0], s[0]
    assert status[bad] == 3 and not want[bad].any() and all(s in (0, 3) for s in status.values())
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    for n in (len(sides), sms // 4, sms // 2 + 1, sms + 1, 2 * sms + 3):
        if n * max(sides) ** 4 > 3e7:
            continue
        idx = [i % len(sides) for i in range(n)]
        got, st = _repeat(cuda, covs, sides, idx)
        for g, s, i in zip(got, st, idx):
            if sides[i] % 2:
                assert s == status[i] and torch.equal(g, want[i]), (n, i, s)
            else:
                assert s == 2
