"""Rendering against the oracle where the kernel's tiles, its launch classes (stamps up to 63 px and larger ones) and the
Moffat integral's branches (step by beta, the folded form above beta = 7 and for tiny arguments) change; max-norm bound of the
rendering test, 1e-5 of the stamp's peak."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu

SIDES = [3, 5, 31, 33, 61, 63, 65, 67, 95, 97, 125, 127]


@pytest.mark.parametrize("kind,beta,fwhm", [("gaussian", 0.0, 0.7), ("moffat", 1.5, 0.7), ("moffat", 3.0, 0.8),
                                            ("moffat", 4.9, 0.6), ("moffat", 5.1, 0.6), ("moffat", 7.5, 0.9),
                                            ("moffat", 3.0, 0.002)])
def test_render_over_classes(cuda, kind, beta, fwhm):
    rng = np.random.default_rng(int(10 * beta))
    n = len(SIDES)
    th = np.column_stack([rng.uniform(2, 3, n), rng.uniform(-0.4, 0.1, n), rng.uniform(-0.4, 0.4, (n, 2)),
                          rng.uniform(-0.5, 0.5, (n, 2))]).astype(np.float32)
    side = torch.from_numpy(np.array(SIDES, np.int32)).to(cuda)
    psf = api.psf_table(kind, np.full(n, fwhm, np.float32), beta, device=cuda)
    out, offs = api.render(torch.from_numpy(th).to(cuda), side, psf)
    out, offs = out.cpu().numpy(), offs.cpu().numpy()
    pk = (O.PSF_GAUSSIAN, float(np.float32(fwhm))) if kind == "gaussian" else (O.PSF_MOFFAT, float(np.float32(fwhm)), beta)
    for i, N in enumerate(SIDES):
        ref = O.render(N, 0.2, pk, th[i].astype(np.float64))
        got = out[offs[i]:offs[i] + N * N].reshape(N, N)
        assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max(), (N, np.abs(got - ref).max() / np.abs(ref).max())
        alone, _ = api.render(torch.from_numpy(th[i:i + 1]).to(cuda), side[i:i + 1],
                              api.psf_table(kind, np.float32(fwhm), beta, device=cuda))
        assert np.array_equal(alone.cpu().numpy()[:N * N], got.ravel()), N
