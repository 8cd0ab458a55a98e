"""A spline with clamped or repeated knots passes through control points; a
span whose Bezier points come from knot insertion keeps such a point as it is,
whatever the size of its neighbours."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("rational", [False, True])
@pytest.mark.parametrize("own_knots", [False, True])
def test_interpolated_points(p, rational, own_knots):
    # two Bezier segments joined by a knot of multiplicity p (own knots), or one
    # (clamped uniform: the spline of p + 1 points)
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(p)
    n, nc = 40, 2 * p + 1 if own_knots else p + 1
    ctrl = rng.uniform(1e9, 4e9, (n, nc, 2)).astype(np.float32)
    at = [0, p, nc - 1] if own_knots else [0, nc - 1]
    ctrl[:, at] = rng.uniform(-1, 1, (n, len(at), 2))
    knots, t = None, [0.0, 1.0]
    if own_knots:
        knots = np.repeat(np.float32([[-1.0, 0.25, 2.0]]), n, 0).repeat([p + 1, p, p + 1], axis=1)
        knots, t = torch.from_numpy(knots).cuda(), [-1.0, 0.25, 2.0]
    x, t = torch.from_numpy(ctrl).cuda(), torch.tensor(t, device="cuda")
    if rational:
        w = rng.uniform(0.5, 2, (n, nc)).astype(np.float32)
        w[:, at] = 1.0
        got = bez.bez_eval_nurbs(x, torch.from_numpy(w).cuda(), p, t, knots=knots)
    else:
        got = bez.bez_eval_bspline(x, p, t, knots=knots)
    assert np.array_equal(got.cpu().numpy(), ctrl[:, at])
