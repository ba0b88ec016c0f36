"""Points of one call: runs of points that share a galaxy are evaluated on one staging, at the edges of the blocks
they are grouped in, over every column-slot class, on FP32 and FP64 stamps."""
import numpy as np
import pytest
import torch

import datagen
import oracle as O
from paper_2604_22048_gb300 import api, synth

pytestmark = pytest.mark.gpu

SIDES = [3, 31, 33, 63, 65, 95, 97, 127]


# runs of one, two, four, five and nine points, across the blocks of four, with an invalid galaxy in between
@pytest.mark.parametrize("top,f64", [(2, False), (4, True), (6, False), (8, False)])
def test_shared_staging_is_the_single_point(cuda, top, f64):
    sides = SIDES[:top]
    truth = synth.draw_ragged(len(sides), seed=11)
    truth.side = np.asarray(sides, dtype=np.int64)
    ds = datagen.make_dataset(truth, 1)
    flat, offs, sd = datagen.pack(ds, np.float64 if f64 else np.float32)
    gi = np.repeat([0, top - 1, 0, -1, 1, top - 1, top - 2, len(sides)], [1, 2, 4, 1, 5, 9, 1, 3]).astype(np.int32)
    rng = np.random.default_rng(top)
    pts = (ds.theta[np.clip(gi, 0, top - 1)] +
           rng.normal(0, [0.02, 0.02, 0.03, 0.03, 0.05, 0.05], (len(gi), 6))).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    args = (t(flat), t(offs), t(sd), api.psf_table("moffat", truth.psf_fwhm.astype(np.float32), truth.psf_beta,
                                                   device=cuda), t(ds.sigma.astype(np.float32)))
    lp, g = [x.cpu().numpy() for x in api.logpost_points(*args, t(gi), t(pts), max_side=max(sides))]
    for i, k in enumerate(gi):
        one, gone = [x.cpu().numpy() for x in api.logpost_points(*args, t(gi[i:i + 1]), t(pts[i:i + 1]),
                                                                 max_side=max(sides))]
        assert np.array_equal(lp[i:i + 1], one, equal_nan=True) and np.array_equal(g[i:i + 1], gone, equal_nan=True)
        if k < 0 or k >= top:
            assert np.isnan(lp[i]) and np.isnan(g[i]).all()
            continue
        N = sides[k]
        ref, gref = O.logpost(N, 0.2, ds.psf[k], ds.stamps[k].astype(flat.dtype).astype(np.float64), 1.0,
                              pts[i].astype(np.float64))
        assert abs(lp[i] - ref) <= 1e-5 * abs(ref), (N, lp[i], ref)
        assert np.abs(g[i] - gref).max() <= 1e-4 * np.abs(gref).max() + 1e-3, (N, g[i], gref)
