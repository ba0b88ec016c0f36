"""Two host threads that call one kernel with small and with large stamps or chains at the same time, straight through the
C calls (which run side by side): each launch keeps its own shared memory, whatever limit the other thread's call sets."""
import ctypes as C
import threading

import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import _ffi as F
from paper_2604_22048_gb300 import api

pytestmark = pytest.mark.gpu
CALLS = 3000


def _ess(cuda, S, stream):
    x = torch.randn((6, 1, 4, S), device=cuda)
    out = torch.empty((1, 6), device=cuda)
    args = [C.c_void_p(x.data_ptr()), 1, 4, S, C.c_void_p(out.data_ptr()), C.c_void_p(0), C.c_void_p(stream.cuda_stream)]
    return (x, out), out, lambda fn=F.lib().bs_chain_ess: fn(*args)


def _galaxy(cuda, side):
    th = torch.tensor([[2.0, -0.2, 0.1, 0.0, 0.1, 0.2]], device=cuda)
    sd = torch.tensor([side], dtype=torch.int32, device=cuda)
    psf = api.psf_table("gaussian", np.array([0.7], np.float32), device=cuda)
    return th, sd, torch.zeros(1, dtype=torch.int64, device=cuda), psf


def _render(cuda, side, stream):
    th, sd, off, psf = _galaxy(cuda, side)
    out = torch.zeros(side * side, device=cuda)
    p = lambda t: C.c_void_p(t.data_ptr())
    args = [1, p(th), C.c_void_p(0), p(off), p(sd), side, p(psf[0]), 1, C.c_float(0.2), p(out),
            C.c_void_p(stream.cuda_stream)]
    return (th, sd, off, psf, out), out, lambda fn=F.lib().bs_render: fn(*args)


def _fit(cuda, side, stream):
    th, sd, off, psf = _galaxy(cuda, side)
    cfg = api.FitConfig(n_chains=1, n_warmup=0, n_samples=1, n_leapfrog=1)
    plan = api.FitPlan(torch.ones(side * side, device=cuda), off, sd, psf, torch.ones(1, device=cuda), th[:, None].contiguous(),
                       cfg, max_side=side)
    args = [C.byref(plan.args), C.byref(plan.out), C.c_void_p(plan.ws.data_ptr()), plan.ws_bytes,
            C.c_void_p(stream.cuda_stream)]
    return plan, plan.samples, lambda fn=F.lib().bs_fit_galaxies: fn(*args)


@pytest.mark.parametrize("make,small,large", [(_ess, 100, 13000), (_render, 65, 127), (_fit, 97, 127)])
def test_two_threads(cuda, make, small, large):
    streams = [torch.cuda.Stream(cuda) for _ in range(2)]
    torch.cuda.synchronize()
    jobs = [make(cuda, size, s) for size, s in zip((small, large), streams)]
    want = []
    for _, out, call in jobs:
        assert call() == 0
        torch.cuda.synchronize()
        want.append(out.clone())
    torch.cuda.synchronize()
    bad = [0, 0]
    go = threading.Barrier(2)

    def work(i, call):
        go.wait()
        for _ in range(CALLS):
            bad[i] += call() != 0

    threads = [threading.Thread(target=work, args=(i, job[2])) for i, job in enumerate(jobs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert bad == [0, 0]
    for (_, out, _), w in zip(jobs, want):
        assert torch.equal(out, w)
