"""GPU parity of the chain kernel with a copy of the chain per lane (in-kernel
draws, 8192 samples and more): run and tile remainders, one segment, many
chains per block, 2D and 3D, output off a 16-byte boundary.

Bounds, a priori (u = 2^-24, M the largest control value): a point rounds 2 d
times in de Casteljau (2 d + 2 in centred Horner, whose coefficients sum to at
most 2^d M), and the local parameter t - k is exact, so |P - P64| <=
(2 d + 2) 2^d u M a component; a length as in test_curve_tile_gpu."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["DECASTELJAU", "HORNER_CENTRED"])
@pytest.mark.parametrize("degree,dim", [(2, 3), (3, 3), (2, 2), (3, 2)])
@pytest.mark.parametrize("out_mode", ["POINTS", "POLYLINE_LENGTH"])
@pytest.mark.parametrize("n,n_seg,n_t", [(3, 1, 8192), (310, 5, 8201), (2, 64, 12345), (1, 33, 65537)])
def test_draws_on_many_segments(variant, degree, dim, out_mode, n, n_seg, n_t):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(degree + 10 * dim + n)
    ctrl = rng.uniform(-1, 1, (n, n_seg * degree + 1, dim)).astype(np.float32)
    t = (np.float32(n_seg) * oracle.hash_t(9, 4, 0, n, n_t).astype(np.float32)).astype(np.float32)
    size = n * n_t * dim if out_mode == "POINTS" else n
    store = torch.full((size + 3,), 9.0, device="cuda")
    out = store[1:1 + size].view((n, n_t, dim) if out_mode == "POINTS" else (n,))
    bez.bez_eval_piecewise(torch.from_numpy(ctrl).cuda(), n_seg, degree, n_t=n_t, variant=bez.Variant[variant],
                           out_mode=bez.OutMode[out_mode], t_mode=bez.TMode.HASH, seed=9, stream_id=4, out=out)
    torch.cuda.synchronize()
    assert store[0] == 9.0 and bool((store[1 + size:] == 9.0).all())
    got = out.cpu().numpy()
    ref = oracle.chain(ctrl, n_seg, degree, t)
    tol = (2 * degree + 2) * 2.0 ** degree * 2.0 ** -24 * np.abs(ctrl).max((1, 2)).astype(np.float64)
    if out_mode == "POINTS":
        assert np.all(np.abs(got - ref) <= tol[:, None, None])
    else:
        L = np.linalg.norm(np.diff(ref, axis=1), axis=2).sum(1)
        assert np.all(np.abs(got - L) <= 2 * n_t * np.sqrt(dim) * tol + n_t * 2.0 ** -23 * L)
