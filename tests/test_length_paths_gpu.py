"""Polyline lengths by path: the size of a call does not change a curve's
length, and no segment is lost or counted twice where the runs of lanes, warps
and blocks join.

With parameters as an array, a curve is sampled at one parameter up to sample j
and at another from there on: its length is one segment, whichever run or join
holds it.  With in-kernel draws every segment counts, and a length is held to a
bound below one segment (asserted).  A priori, u = 2^-24: a segment's difference,
squares and approximate root round by at most 6 u of it, a sum of depth D by D u,
and each end moves by at most a point's error, (2 d + 2) 2^d u M a component (see
test_curve_tile_gpu), so |L - L64| <= (6 + D) u L + 2 n sqrt(dim) (2 d + 2) 2^d u M."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.mark.parametrize("variant", ["HORNER", "HORNER_CENTRED", "BERNSTEIN", "DECASTELJAU", "SEILER"])
@pytest.mark.parametrize("d, dim", [(1, 1), (3, 3), (2, 2), (4, 3), (4, 4), (5, 3), (6, 2), (7, 4)])
def test_lengths_do_not_depend_on_the_call(variant, d, dim):
    # 2 curves, then fewer lanes a run for more of them, then a lane a run
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    g = torch.Generator(device="cuda").manual_seed(10 * d + dim)
    for n_t in (1, 2, 9, 31, 33, 64, 65, 100, 128, 130, 255, 256, 400, 512, 601, 1024, 1030, 2047, 4096, 4100, 9000):
        sizes = [2, 700, 2500, 6000, 12_000] if n_t <= 1024 else [2, 1500, 5000]
        ctrl = torch.rand((sizes[-1], d + 1, dim), generator=g, device="cuda") * 2 - 1
        t = torch.rand(n_t, generator=g, device="cuda")
        for mode in ("SHARED", "UNIFORM", "HASH"):
            first = None
            for n in sizes:
                store = torch.full((n + 2,), -1.0, device="cuda")
                bez.bez_eval(ctrl[:n], t if mode == "SHARED" else None, n_t=n_t, variant=bez.Variant[variant],
                             t_mode=bez.TMode[mode], out_mode=bez.OutMode.POLYLINE_LENGTH, seed=7, stream_id=3,
                             out=store[1:-1])
                assert store[0] == -1.0 and store[-1] == -1.0
                first = store[1:3].clone() if first is None else first
                assert torch.equal(store[1:3], first), (n, n_t, mode)


def _jumps(n_t, lo, hi, copies):
    """t [copies (n_t - 1)][n_t]: lo up to sample j, hi from there on, for every j."""
    j = np.arange(1, n_t)
    return np.tile(np.where(np.arange(n_t)[None] < j[:, None], np.float32(lo), np.float32(hi)), (copies, 1))


@pytest.mark.parametrize("variant", ["HORNER_CENTRED", "DECASTELJAU"])
@pytest.mark.parametrize("d, dim", [(3, 3), (5, 2), (2, 4)])
@pytest.mark.parametrize("n_t, copies", [(2, 3), (17, 1), (33, 1), (33, 600), (64, 1), (100, 1), (129, 1), (129, 80),
                                         (256, 1), (513, 1), (513, 20), (1025, 1), (1025, 8)])
def test_every_segment_once(variant, d, dim, n_t, copies):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(d + n_t)
    t = _jumps(n_t, 0.125, 0.875, copies)
    b = rng.uniform(0, 1, (1, d + 1, dim)).astype(np.float32) + np.arange(d + 1, dtype=np.float32)[None, :, None]
    ctrl = np.broadcast_to(b, (len(t), d + 1, dim)).copy()
    got = bez.bez_eval(torch.from_numpy(ctrl).cuda(), torch.from_numpy(t).cuda(), variant=bez.Variant[variant],
                       out_mode=bez.OutMode.POLYLINE_LENGTH).cpu().numpy()
    ends = oracle.bezier(b, np.float32([0.125, 0.875]))
    L = np.linalg.norm(ends[0, 1] - ends[0, 0])
    assert np.all(np.abs(got - L) <= 6 * U * L + 2 * np.sqrt(dim) * (2 * d + 2) * 2.0 ** d * U * b.max())


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("rational", [False, True])
@pytest.mark.parametrize("n_t, copies", [(2, 2), (31, 1), (32, 1), (33, 70), (65, 1), (200, 1)])
def test_every_segment_once_splines(p, rational, n_t, copies):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(p + n_t)
    nc = 11
    t = _jumps(n_t, 0.1, 0.9, copies)
    b = rng.uniform(0, 1, (1, nc, 3)).astype(np.float32) + np.arange(nc, dtype=np.float32)[None, :, None]
    w = rng.uniform(0.5, 2, (1, nc)).astype(np.float32) if rational else None
    ctrl = torch.from_numpy(np.broadcast_to(b, (len(t), nc, 3)).copy()).cuda()
    kw = dict(out_mode=bez.OutMode.POLYLINE_LENGTH)
    if rational:
        wt = torch.from_numpy(np.broadcast_to(w, (len(t), nc)).copy()).cuda()
        got = bez.bez_eval_nurbs(ctrl, wt, p, torch.from_numpy(t).cuda(), **kw)
    else:
        got = bez.bez_eval_bspline(ctrl, p, torch.from_numpy(t).cuda(), **kw)
    ends = oracle.bspline(b, p, np.float32([0.1, 0.9]), weights=w)
    L = np.linalg.norm(ends[0, 1] - ends[0, 0])
    # points: 3 p + 4 roundings of values up to M (homogeneous ones up to 2 M, over a weight of 0.5 and more)
    tol = (3 * p + 4) * U * b.max() * (8 if rational else 1)
    assert np.all(np.abs(got.cpu().numpy() - L) <= 6 * U * L + 2 * np.sqrt(3) * tol)


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("mode", ["UNIFORM", "HASH"])
@pytest.mark.parametrize("n, n_t", [(5, 1), (3, 31), (9, 32), (7, 33), (2, 1000)])  # (1000 steps of a grid are too short)
def test_spline_lengths(p, mode, n, n_t):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(p + n_t)
    ctrl = rng.uniform(-1, 1, (n, 9, 3)).astype(np.float32)
    t = oracle.grid(n_t).astype(np.float32) if mode == "UNIFORM" else oracle.hash_t(7, 3, 0, n, n_t)
    got = bez.bez_eval_bspline(torch.from_numpy(ctrl).cuda(), p, n_t=n_t, t_mode=bez.TMode[mode], seed=7, stream_id=3,
                               out_mode=bez.OutMode.POLYLINE_LENGTH).cpu().numpy()
    seg = np.linalg.norm(np.diff(oracle.bspline(ctrl, p, t), axis=1), axis=2)
    L = seg.sum(1)
    # local parameters round once more, which moves a point by at most 2 p M u 6 (spans) more
    tol = (6 + n_t / 32 + 8) * U * L + 2 * n_t * np.sqrt(3) * (15 * p + 4) * U
    assert n_t < 32 or (mode == "UNIFORM" and n_t > 100) or np.all(tol < 0.5 * seg.mean(1))
    assert np.all(np.abs(got - L) <= tol)


@pytest.mark.parametrize("d, dim", [(3, 3), (1, 1), (2, 2), (4, 3), (3, 4), (5, 3), (6, 2)])
@pytest.mark.parametrize("n, n_t", [(40, 40), (40, 64), (40, 131), (40, 256), (20, 1000), (20, 1024), (7, 1030), (9, 2048),
                                    (3, 4099), (3000, 100)])
def test_draws(d, dim, n, n_t):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(d + n_t)
    ctrl = rng.uniform(-1, 1, (n, d + 1, dim)).astype(np.float32)
    got = bez.bez_eval(torch.from_numpy(ctrl).cuda(), n_t=n_t, t_mode=bez.TMode.HASH, seed=7, stream_id=3,
                       out_mode=bez.OutMode.POLYLINE_LENGTH).cpu().numpy()
    seg = np.linalg.norm(np.diff(oracle.bezier(ctrl, oracle.hash_t(7, 3, 0, n, n_t)), axis=1), axis=2)
    L = seg.sum(1)
    tol = (6 + 32 + 16) * U * L + 2 * n_t * np.sqrt(dim) * (2 * d + 2) * 2.0 ** d * U * np.abs(ctrl).max((1, 2))
    assert np.median(tol / seg.mean(1)) < (0.5 if n_t < 2000 else 2)  # (longer curves: of the 16 joins and more)
    assert np.all(np.abs(got - L) <= tol)


@pytest.mark.parametrize("variant", ["DECASTELJAU", "HORNER_CENTRED"])
@pytest.mark.parametrize("degree, dim", [(2, 3), (3, 3), (2, 2), (3, 2)])
@pytest.mark.parametrize("n, n_seg, n_t", [(40, 5, 8192), (40, 9, 8201), (9, 64, 12345), (3, 33, 65537)])
def test_chains_at_draws(variant, degree, dim, n, n_seg, n_t):
    # a run of n_t / 512 samples in two halves, then 9 levels of lanes and warps
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(degree + n_t)
    ctrl = rng.uniform(-1, 1, (n, n_seg * degree + 1, dim)).astype(np.float32)
    t = (np.float32(n_seg) * oracle.hash_t(9, 4, 0, n, n_t).astype(np.float32)).astype(np.float32)
    got = bez.bez_eval_piecewise(torch.from_numpy(ctrl).cuda(), n_seg, degree, n_t=n_t, variant=bez.Variant[variant],
                                 out_mode=bez.OutMode.POLYLINE_LENGTH, t_mode=bez.TMode.HASH, seed=9,
                                 stream_id=4).cpu().numpy()
    seg = np.linalg.norm(np.diff(oracle.chain(ctrl, n_seg, degree, t), axis=1), axis=2)
    L = seg.sum(1)
    tol = (6 + n_t / 1024 + 16) * U * L + 2 * n_t * np.sqrt(dim) * (2 * degree + 2) * 2.0 ** degree * U
    assert np.all(tol < (4 if n_t > 20_000 else 1) * seg.mean(1))
    assert np.all(np.abs(got - L) <= tol)
