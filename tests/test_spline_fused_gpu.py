"""GPU parity of the one-kernel spline path (degrees 1..5 whose spans fit in
shared memory) at the edges of its blocks: curves per block from many to one,
samples cut into ranges, samples shorter and longer than a warp's tile, output
off a 16-byte boundary, and values near the end of the FP32 range.

Bound, a priori (u = 2^-24, M the largest control value): the span points are
rounded once, de Casteljau rounds 2 p times, tau once with |dC/dtau| <= 2 p M,
so |P - P64| <= (6 p + 4) u M; homogeneous coordinates are at most 2 M with
weights in [0.5, 2], and the quotient by a weight >= 0.5 makes it 10 times that."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

#         n curves, n_ctrl over degree + 1, samples
SHAPES = [(1, 0, 1), (40, 0, 5), (200, 1, 33), (3000, 2, 17), (65, 30, 129), (3, 59, 700), (2, 200, 5000),
          (1500, 11, 130)]


def _knots(rng, n, n_ctrl, p):
    gaps = rng.uniform(0.25, 1.25, (n, n_ctrl - p))
    inner = (np.cumsum(gaps, 1) / gaps.sum(1, keepdims=True))[:, :-1]
    return np.concatenate([np.zeros((n, p + 1)), inner, np.ones((n, p + 1))], 1).astype(np.float32)


def _run(torch, ctrl, p, t, w, U, out=None):
    from paper_2603_15447_gb300 import bez

    def dev(x):
        return None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()
    if w is None:
        return bez.bez_eval_bspline(dev(ctrl), p, dev(t), knots=dev(U), out=out)
    return bez.bez_eval_nurbs(dev(ctrl), dev(w), p, dev(t), knots=dev(U), out=out)


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("rational", [False, True])
@pytest.mark.parametrize("knots", [False, True])
def test_block_edges(p, rational, knots):
    torch = need_gpu()
    for i, (n, more, n_t) in enumerate(SHAPES):
        rng = np.random.default_rng(1000 * p + i)
        dim, n_ctrl = 1 + (i + p) % 4, p + 1 + more
        ctrl = rng.uniform(-1, 1, (n, n_ctrl, dim)).astype(np.float32)
        w = rng.uniform(0.5, 2, (n, n_ctrl)).astype(np.float32) if rational else None
        U = _knots(rng, n, n_ctrl, p) if knots else None
        t = rng.uniform(0, 1, (n, n_t) if i % 2 else n_t).astype(np.float32)
        store = torch.full((n * n_t * dim + 3,), 9.0, device="cuda")
        out = store[1:1 + n * n_t * dim].view(n, n_t, dim)
        got = _run(torch, ctrl, p, t, w, U, out).cpu().numpy()
        assert store[0] == 9.0 and bool((store[1 + n * n_t * dim:] == 9.0).all())
        ref = oracle.bspline(ctrl, p, t, weights=w, knots=U)
        tol = (6 * p + 4) * 2.0 ** -24 * np.abs(ctrl).max((1, 2)).astype(np.float64) * (10 if rational else 1)
        assert np.all(np.abs(got - ref) <= tol[:, None, None]), (n, n_ctrl, n_t, dim)


@pytest.mark.parametrize("p", [2, 3, 5])
def test_values_at_the_end_of_the_range(p):
    """Differences of control points that overflow FP32 are taken in FP64; an
    infinite control point reaches the spans that use it and no other."""
    torch = need_gpu()
    rng = np.random.default_rng(p)
    clean = rng.uniform(-1, 1, (5, 20, 3)).astype(np.float32)
    t = ((np.arange(200, dtype=np.float32) + np.float32(0.5)) / np.float32(200)).astype(np.float32)
    big = (clean * np.float32(3.0e38)).astype(np.float32)
    got = _run(torch, big, p, t, None, None).cpu().numpy().astype(np.float64)
    ref = oracle.bspline(big, p, t)
    assert np.all(np.abs(got - ref) <= (6 * p + 4) * 2.0 ** -24 * 3.0e38)
    bad = clean.copy()
    bad[2, 10, 1] = np.inf
    got = _run(torch, bad, p, t, None, None).cpu().numpy()
    want = _run(torch, clean, p, t, None, None).cpu().numpy()
    span = np.minimum((t.astype(np.float64) * (20 - p)).astype(int), 20 - p - 1)
    uses = (span <= 10) & (span + p >= 10)
    assert not np.isfinite(got[2, uses, 1]).any()
    got[2, uses, 1] = want[2, uses, 1]
    # the same spans, extracted in FP64 for this curve and in float-float for the clean one
    assert np.all(np.abs(got[2] - want[2]) <= (6 * p + 4) * 2.0 ** -24)
    got[2] = want[2]
    np.testing.assert_array_equal(got, want)
