"""One curve at the largest sample count: it is cut into ranges like any other
long curve (a warp alone would take seconds)."""
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_t", [2 ** 31 - 1, 2 ** 31 - 300])
def test_longest_curve(n_t):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    ctrl = torch.tensor([[[0.0], [1.0]]], device="cuda")
    out = torch.empty((1, n_t, 1), device="cuda")
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    begin.record()
    bez.bez_eval(ctrl, n_t=n_t, t_mode=bez.TMode.UNIFORM, out=out)
    end.record()
    torch.cuda.synchronize()
    assert begin.elapsed_time(end) < 1000
    j = torch.tensor([0, 1, 255, 256, 1 << 20, 1 << 30, n_t - 257, n_t - 2, n_t - 1], device="cuda")
    want = j.float() / torch.tensor(float(n_t - 1), device="cuda")      # x = t, up to the centred form's two roundings
    assert bool(((out[0, j, 0] - want).abs() <= 2.0 ** -23).all())
