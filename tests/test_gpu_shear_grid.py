"""The one-point pass over rows that do not go through tiles (K not a multiple of 4, rows off a 16-byte boundary) fills
the GPU: its kernels hold three CTAs per SM, with per-sample offsets and without, and each CTA leaves its four partial sums at
the front of the workspace."""
import pytest
import torch

from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family", [0, 1])
@pytest.mark.parametrize("offsets", [False, True])
@pytest.mark.parametrize("K,shift", [(7, 0), (99, 0), (8, 1)])
def test_scalar_rows_fill_the_gpu(cuda, family, offsets, K, shift):
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    n = 32 * 4 * sms

    def rows():
        x = 0.1 * torch.randn(n * K + shift, device=cuda)
        return x[shift:].reshape(n, K)

    plan = api.ShearPlan(rows(), rows(), rows() if offsets else None, family=family, trunc_r=0.7)
    plan.ws.fill_(255)
    plan.loglike(0.02, -0.01, 0.2)
    words = plan.ws.view(torch.int64)
    written = (words != -1).cpu()
    ctas = int((~written).nonzero()[0]) // 4 if not bool(written.all()) else len(written) // 4
    assert ctas >= 3 * sms, (ctas, sms)
