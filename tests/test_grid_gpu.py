"""GPU parity of the general grid kernel (any degrees, any dimension, surfaces
as one-slab volumes) at the edges of its blocks of 32 rows and tiles of 128
points, with the output off a 16-byte boundary and half-precision storage.

Bound, a priori (u = 2^-24, M the largest control value): a Bernstein value is
a product of at most d + 2 rounded factors, each of the two or three
contractions sums d + 1 terms of a partition of unity, so
|P - P64| <= sum over the axes of (2 d + 4) u M."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _check(torch, ctrl, grid, half):
    from paper_2603_15447_gb300 import bez
    c = torch.from_numpy(ctrl).cuda()
    if half:
        c = c.half()
        ctrl = c.float().cpu().numpy()
    n, dim = ctrl.shape[0], ctrl.shape[-1]
    size = n * int(np.prod(grid)) * dim
    store = torch.full((size + 3,), 9.0, device="cuda")
    out = store[1:1 + size].view(n, *grid, dim)
    if len(grid) == 2:
        bez.bez_eval_surface(c, *grid, out=out)
        ref = oracle.surface(ctrl, *grid)
    else:
        bez.bez_eval_volume(c, *grid, out=out)
        ref = oracle.volume(ctrl, *grid)
    torch.cuda.synchronize()
    assert store[0] == 9.0 and bool((store[1 + size:] == 9.0).all())
    tol = sum(2 * (d - 1) + 4 for d in ctrl.shape[1:-1]) * 2.0 ** -24 * np.abs(ctrl).max()
    assert np.abs(out.cpu().numpy() - ref).max() <= tol


@pytest.mark.parametrize("du,dv,dim", [(3, 3, 3), (1, 2, 1), (4, 3, 2), (2, 5, 4), (7, 7, 3)])
@pytest.mark.parametrize("nu,nv", [(1, 1), (32, 4), (33, 31), (3, 129), (97, 7)])
@pytest.mark.parametrize("half", [False, True])
def test_surfaces(du, dv, dim, nu, nv, half):
    torch = need_gpu()
    rng = np.random.default_rng(100 * du + 10 * dv + nu)
    _check(torch, rng.uniform(-1, 1, (9, du + 1, dv + 1, dim)).astype(np.float32), (nu, nv), half)


@pytest.mark.parametrize("d,dim", [((3, 3, 3), 3), ((1, 2, 3), 2), ((2, 1, 5), 1), ((3, 4, 2), 4), ((7, 7, 7), 4)])
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 33, 5), (5, 3, 40), (20, 24, 28)])
def test_volumes(d, dim, grid):
    torch = need_gpu()
    rng = np.random.default_rng(sum(d) + grid[1])
    _check(torch, rng.uniform(-1, 1, (5, d[0] + 1, d[1] + 1, d[2] + 1, dim)).astype(np.float32), grid, False)
