"""GPU parity of the adjoint for curves far from the origin.  C' is a sum of
differences of control points, so the bound on dL/dt (test_grad_gpu: O(d)
roundings of g . C', scaled by the largest difference) holds wherever the
curve lies; so does the one on dL/dP, which no coordinate enters."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_grad_gpu import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("dim", [1, 2, 3, 4])
@pytest.mark.parametrize("offset", [-10.0, 1e3, 1e5])
def test_offset_curves(d, dim, offset):
    torch = need_gpu()
    rng = np.random.default_rng(100 * d + dim)
    B, n_t = 101, 70
    ctrl = (offset + rng.uniform(-1, 1, (B, d + 1, dim))).astype(np.float32)
    t = rng.uniform(0, 1, (B, n_t)).astype(np.float32)
    _check(torch, ctrl, t, rng.normal(size=(B, n_t, dim)).astype(np.float32))
