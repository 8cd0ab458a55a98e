"""Centred Horner of degree 5..7 near the end of the FP32 range: the terms of
its coefficients leave the range where the coefficients themselves do not."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [5, 6, 7])
@pytest.mark.parametrize("dim", [1, 2, 3, 4])
def test_large_points(d, dim):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(d)
    ctrl = (2e38 * (1 + 1e-4 * rng.uniform(-1, 1, (40, d + 1, dim)))).astype(np.float32)
    t = np.linspace(0, 1, 70, dtype=np.float32)
    got = bez.bez_eval(torch.from_numpy(ctrl).cuda(), torch.from_numpy(t).cuda(), variant=bez.Variant.HORNER_CENTRED)
    ref = oracle.bezier(ctrl, t)
    # the coefficients rounded once (those of order >= 1 are 1e-4 of the points) and d fused steps
    assert np.all(np.abs(got.cpu().numpy() - ref) <= 4 * 2.0 ** -24 * np.abs(ref))
