"""GPU parity of the fixed-degree adjoint kernels over dimensions and sample
counts around a warp's 64-sample step, with the tolerances of test_grad_gpu
(each term with O(d) roundings, summed per lane and over the warp)."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_grad_gpu import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("dim", [1, 2, 3, 4])
@pytest.mark.parametrize("rational", [False, True])
def test_dims_and_sample_counts(d, dim, rational):
    torch = need_gpu()
    rng = np.random.default_rng(100 * d + 10 * dim + rational)
    for n_t in (1, 31, 33, 64, 65, 200):
        B = 41
        ctrl = rng.uniform(-1, 1, (B, d + 1, dim)).astype(np.float32)
        w = rng.uniform(0.5, 2, (B, d + 1)).astype(np.float32) if rational else None
        t = rng.uniform(0, 1, n_t if n_t == 65 else (B, n_t)).astype(np.float32)
        t[..., 0] = 1.25                                  # clamped: zero dL/dt
        _check(torch, ctrl, t, rng.normal(size=(B, n_t, dim)).astype(np.float32), w)
