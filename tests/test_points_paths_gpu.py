"""The paths of curve points by the size of a call (a thread per sample or per
2, 4, 8 of them; tiles of several curves a warp): a curve's points are the same
to the last bit whatever the call, its first calls compared with the oracle by
test_curve_tile_gpu."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

# one thread per sample, then each larger call on the next path
SIZES = {8: (41, 100_003, 130_000), 63: (41, 9001, 16_000), 257: (41, 1951, 5801, 11_601, 16_001), 70_001: (1, 30, 60)}


@pytest.mark.parametrize("variant", ["HORNER", "HORNER_CENTRED", "BERNSTEIN", "DECASTELJAU", "SEILER"])
@pytest.mark.parametrize("d, dim", [(1, 1), (2, 3), (3, 3), (3, 2), (4, 4), (5, 2), (7, 3)])
def test_points_do_not_depend_on_the_call(variant, d, dim):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    g = torch.Generator(device="cuda").manual_seed(10 * d + dim)
    for k, (n_t, sizes) in enumerate(SIZES.items()):
        ctrl = torch.rand((sizes[-1], d + 1, dim), generator=g, device="cuda") * 2 - 1
        if k == 1:
            ctrl = ctrl.half()
        t = torch.rand(n_t, generator=g, device="cuda")
        for mode in ("SHARED", "UNIFORM", "HASH"):
            kw = dict(n_t=n_t, variant=bez.Variant[variant], t_mode=bez.TMode[mode], seed=7, stream_id=3)
            m, want = sizes[0], None
            for n in sizes:
                store = torch.full((n * n_t * dim + 3,), 9.0, device="cuda")
                out = store[1:-2].view(n, n_t, dim)       # 4 bytes past a 16-byte boundary, guards on both sides
                bez.bez_eval(ctrl[:n], t if mode == "SHARED" else None, out=out, **kw)
                assert store[0] == 9.0 and bool((store[-2:] == 9.0).all()) and bool(torch.isfinite(out).all())
                want = out[:m].clone() if want is None else want
                assert torch.equal(out[:m], want), (n, n_t, mode)


def test_own_parameters_outside_the_interval():
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    g = torch.Generator(device="cuda").manual_seed(1)
    ctrl = torch.rand((16_001, 4, 3), generator=g, device="cuda")
    t = torch.rand((16_001, 256), generator=g, device="cuda") * 1.5 - 0.25
    t[:, 5] = float("nan")
    big = bez.bez_eval(ctrl, t)
    for n in (3, 2000, 6000, 11_000):
        assert torch.equal(torch.nan_to_num(bez.bez_eval(ctrl[:n], t[:n]), nan=9.0), torch.nan_to_num(big[:n], nan=9.0))
    assert bool(torch.isnan(big[:, 5]).all()) and bool(torch.equal(big[:, t[0] < 0][0], big[0, t[0] < 0]))
    low = t < 0
    assert torch.equal(big[low], ctrl[:, None, 0].expand(-1, 256, -1)[low]) or bool(
        ((big - ctrl[:, None, 0])[low].abs() <= 8 * 2.0 ** -24 * 8).all())   # (2 d + 2) 2^-24 2^d M
