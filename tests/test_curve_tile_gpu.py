"""GPU parity of the fixed-degree tile kernels (points and lengths of any
dimension, several curves per warp) at the edges of their tiles: sample counts
around the lanes-per-curve steps, one curve more than a warp's, curves cut
into ranges, an output that starts off a 16-byte boundary.

Bounds, a priori.  A component of a point: the centred power coefficients sum
to at most sum_m binom(d, m) 2^m M 2^-m = 2^d M at |u| <= 1/2 (M the curve's
largest control value), Horner and de Casteljau round 2 d times and the
coefficients once, so |P - P64| <= (2 d + 2) 2^-24 2^d M.  A length: each of
the n - 1 segments moves by at most twice a point's error, and a sum of n terms
rounds by at most n 2^-23 of itself (the square root is approximate)."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (9, 8), (17, 33), (33, 65), (5, 129), (3, 257), (2, 5000), (20011, 40)]


def _case(d, dim, n, n_t, mode, seed):
    rng = np.random.default_rng(seed)
    ctrl = rng.uniform(-1, 1, (n, d + 1, dim)).astype(np.float32)
    if mode == "PER_CURVE":
        t = rng.uniform(0, 1, (n, n_t)).astype(np.float32)
    elif mode == "UNIFORM":
        t = oracle.grid(n_t).astype(np.float32)
    else:
        t = oracle.hash_t(7, 3, 0, n, n_t)
    return ctrl, t


@pytest.mark.parametrize("variant", ["HORNER_CENTRED", "DECASTELJAU"])
@pytest.mark.parametrize("d,dim", [(1, 2), (3, 1), (3, 2), (3, 3), (2, 4), (5, 2), (7, 4), (6, 3)])
@pytest.mark.parametrize("out_mode", ["POINTS", "POLYLINE_LENGTH"])
def test_tile_edges(variant, d, dim, out_mode):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    for k, (n, n_t) in enumerate(SHAPES):
        mode = ("PER_CURVE", "UNIFORM", "HASH")[k % 3]
        ctrl, t = _case(d, dim, n, n_t, mode, 10 * d + dim + k)
        dt = torch.from_numpy(t).cuda() if mode == "PER_CURVE" else None
        size = n * n_t * dim if out_mode == "POINTS" else n
        shape = (n, n_t, dim) if out_mode == "POINTS" else (n,)
        store = torch.full((size + 3,), 9.0, device="cuda")
        out = store[1:1 + size].view(shape)   # 4 bytes past a 16-byte boundary, a guard on both sides
        bez.bez_eval(torch.from_numpy(ctrl).cuda(), dt, n_t=n_t, variant=bez.Variant[variant],
                     out_mode=bez.OutMode[out_mode], t_mode=bez.TMode[mode], seed=7, stream_id=3, out=out)
        torch.cuda.synchronize()
        assert store[0] == 9.0 and bool((store[1 + size:] == 9.0).all())
        got = out.cpu().numpy()
        ref = oracle.bezier(ctrl, t)
        tol = (2 * d + 2) * 2.0 ** -24 * 2.0 ** d * np.abs(ctrl).max((1, 2)).astype(np.float64)
        if out_mode == "POINTS":
            assert np.all(np.abs(got - ref) <= tol[:, None, None]), (n, n_t, mode)
        else:
            L = np.linalg.norm(np.diff(ref, axis=1), axis=2).sum(1)
            assert np.all(np.abs(got - L) <= 2 * n_t * np.sqrt(dim) * tol + n_t * 2.0 ** -23 * L), (n, n_t, mode)


@pytest.mark.parametrize("d", [3, 5, 7])
def test_infinite_and_nan_control_points_stay_with_their_curve(d):
    """A non-finite control value reaches its own curve and component only."""
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(d)
    clean = rng.uniform(-1, 1, (40, d + 1, 2)).astype(np.float32)
    ctrl = clean.copy()
    ctrl[3, 1, 0], ctrl[11, d, 1] = np.inf, np.nan
    t = torch.from_numpy(rng.uniform(0.1, 0.9, 20).astype(np.float32)).cuda()
    got = bez.bez_eval(torch.from_numpy(ctrl).cuda(), t).cpu().numpy()
    want = bez.bez_eval(torch.from_numpy(clean).cuda(), t).cpu().numpy()
    assert not np.isfinite(got[3, :, 0]).any() and np.isnan(got[11, :, 1]).all()
    got[3, :, 0], got[11, :, 1] = want[3, :, 0], want[11, :, 1]
    np.testing.assert_array_equal(got, want)
