"""Offsets of packed stamps against their definition: each stamp starts where the one before ends, rounded up."""
import numpy as np
import pytest

from paper_2604_22048_gb300.api import pack_stamps


@pytest.mark.parametrize("align", [1, 4, 16])
@pytest.mark.parametrize("sides", [[], [25], [3], [25, 31], [101, 3, 53, 53, 27]])
@pytest.mark.parametrize("kind", [list, np.int32, np.int64])
def test_offsets(sides, align, kind):
    offs, total = pack_stamps(list(sides) if kind is list else np.array(sides, dtype=kind), align)
    want, at = [], 0
    for s in sides:
        want.append(at)
        at += -(-s * s // align) * align
    assert offs.dtype == np.int64 and offs.tolist() == want
    assert isinstance(total, int) and total == at
