"""Batches of shear points: 16 and more are finalized together and their results copied to the host in stages of up to 512;
every count around those, on the host and on the device, has the bits of the same points four at a time, also in the
smallest workspace the call takes, which holds one pass at a time."""
import ctypes as C
import re

import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import _ffi as F
from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu


def _plan(cuda, K, weighted=False):
    rng = np.random.default_rng(K)
    e1, e2 = rng.normal(0, 0.2, (2, 300, K)).astype(np.float32).clip(-0.6, 0.6)
    w = rng.uniform(0, 2, 300).astype(np.float32) if weighted else None
    return api.ShearPlan(torch.from_numpy(e1).to(cuda), torch.from_numpy(e2).to(cuda), weights=w)


def _points(n):
    t = np.arange(n)
    return np.column_stack([0.03 * np.sin(t), 0.03 * np.cos(1.7 * t), 0.05 + 0.3 * (t % 7) / 7])


@pytest.mark.parametrize("K,weighted", [(64, False), (37, True)])
def test_counts(cuda, K, weighted):
    plan, pts = _plan(cuda, K, weighted), _points(531)
    four = np.concatenate([plan.loglike_multi(pts[i:i + 4]) for i in range(0, 531, 4)])
    for n in (15, 16, 17, 30, 31, 32, 512, 513, 531):
        assert np.array_equal(plan.loglike_multi(pts[:n]), four[:n]), n
        assert np.array_equal(plan.loglike_multi(pts[:n], host=False).cpu().numpy(), four[:n]), n


def test_smallest_workspace(cuda):
    plan, pts = _plan(cuda, 64), _points(33)
    want = plan.loglike_multi(pts)
    lib, p = F.lib(), lambda a: a.ctypes.data_as(C.c_void_p)
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    out = np.zeros((33, 4))

    def call(nbytes):
        return lib.bs_shear_loglike_multi(C.byref(plan.data), 33, p(pts), p(out), 1, C.c_void_p(plan.ws.data_ptr()), nbytes,
                                          stream)

    assert call(8) != 0
    need = int(re.search(r"workspace of (\d+) bytes", lib.bs_last_error().decode()).group(1))
    assert call(need - 1) != 0 and need < plan.ws_bytes
    for nbytes in (need, need + 8 * 63, 2 * need, 4 * need, plan.ws_bytes):
        out[:] = 0
        assert call(nbytes) == 0
        assert np.array_equal(out, want), nbytes


def test_launches_of_a_batch(cuda):
    plan = _plan(cuda, 64)
    before = api.kernel_launches()
    plan.loglike_multi(_points(16))
    assert api.kernel_launches() - before == 5          # four passes, one finalize
