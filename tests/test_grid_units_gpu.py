"""Grids cut into units by the size of a call: a patch's points are the same to
the last bit alone, among a few and among many (32 rows a unit); alone they are
compared with the oracle by test_grid_gpu."""
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _check(torch, call, ctrl, shape, sizes):
    want = None
    for n in sizes:
        store = torch.full((n * int(torch.tensor(shape).prod()) + 2,), 9.0, device="cuda")
        out = store[1:-1].view(n, *shape)              # 4 bytes past a 16-byte boundary, guards on both sides
        call(ctrl[:n], out)
        assert store[0] == 9.0 and store[-1] == 9.0
        want = out[0].clone() if want is None else want
        assert torch.equal(out[0], want) and torch.equal(out[n - 1], out[n - 1].nan_to_num(nan=9.0))


@pytest.mark.parametrize("du, dv, dim", [(2, 2, 3), (5, 4, 1), (3, 3, 4), (1, 7, 2)])
@pytest.mark.parametrize("nu, nv", [(1, 1), (4, 4), (33, 31), (16, 256), (96, 5), (256, 3)])
def test_surfaces(du, dv, dim, nu, nv):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    sizes = (1, 7, 150, 700, 5000)
    ctrl = torch.rand((sizes[-1], du + 1, dv + 1, dim), device="cuda") * 2 - 1
    _check(torch, lambda c, o: bez.bez_eval_surface(c, nu, nv, out=o), ctrl, (nu, nv, dim), sizes)


@pytest.mark.parametrize("d, dim", [((3, 3, 3), 3), ((1, 2, 5), 1), ((2, 1, 1), 4)])
@pytest.mark.parametrize("grid", [(1, 1, 1), (4, 33, 5), (3, 40, 32), (20, 7, 9)])
def test_volumes(d, dim, grid):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    sizes = (1, 7, 150, 2500)
    ctrl = torch.rand((sizes[-1], d[0] + 1, d[1] + 1, d[2] + 1, dim), device="cuda") * 2 - 1
    _check(torch, lambda c, o: bez.bez_eval_volume(c, *grid, out=o), ctrl, (*grid, dim), sizes)
