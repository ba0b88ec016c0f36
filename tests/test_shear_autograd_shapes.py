"""The shapes of the parameters that ShearLogLike takes: a vector of three, or a column; a row is refused."""
import numpy as np
import pytest
import torch

from paper_2604_22048_gb300 import api


class _Plan:
    def loglike(self, g1, g2, alpha, *, host):
        assert all(isinstance(x, float) for x in (g1, g2, alpha)) and host
        return np.array([g1 + 10.0 * g2 + 100.0 * alpha, 1.0, 10.0, 100.0])


@pytest.mark.parametrize("shape", [(3,), (3, 1), (3, 1, 1)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.int64])
def test_vectors_and_columns(shape, dtype):
    v = api.ShearLogLike.apply(torch.tensor([1, 2, 3], dtype=dtype).reshape(shape), _Plan())
    assert v.shape == () and v.dtype == torch.float64 and float(v) == 321.0


@pytest.mark.parametrize("shape", [(1, 3), (2,), (4,), (3, 2)])
def test_other_shapes_are_refused(shape):
    with pytest.raises((ValueError, RuntimeError, TypeError)):
        api.ShearLogLike.apply(torch.zeros(shape), _Plan())


def test_gradient_of_a_vector():
    x = torch.tensor([0.1, 0.2, 0.3], dtype=torch.float64, requires_grad=True)
    (g,) = torch.autograd.grad(api.ShearLogLike.apply(x, _Plan()), x)
    assert g.tolist() == [1.0, 10.0, 100.0]
