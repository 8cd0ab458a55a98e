"""Overlapping launches of one large batch plan without a graph: each stream's
launch is complete by itself, so work ordered after the second stream alone
sees every sample."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_launches_on_two_streams():
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    n, n_s, dim = 1000, 61000, 2                       # 6.1e7 samples
    i = np.arange(n)
    kind = (i % 3).astype(np.int32)
    n_ctrl = np.where(kind == 0, 4, 9)
    rng = np.random.default_rng(5)
    off = np.concatenate([[0], np.cumsum(n_ctrl)])
    desc = bez.descriptors(kind, np.full(n, 3), n_ctrl, np.full(n, n_s), off[:-1] * dim, off[:-1], i * n_s * dim)
    ctrl = torch.from_numpy(rng.uniform(-1, 1, off[-1] * dim).astype(np.float32)).cuda()
    wts = torch.from_numpy(rng.uniform(0.5, 2, off[-1]).astype(np.float32)).cuda()
    out = torch.empty(n * n_s * dim, device="cuda")
    batch = bez.Batch(desc, dim, ctrl, wts, out, use_graph=False)
    assert batch.config()["schedule"] == 0             # a queue would be shared by both launches
    batch.launch()
    want = out.clone()
    assert torch.isfinite(want).all()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        out.fill_(float("nan"))
        torch.cuda.synchronize()
        batch.launch(stream=s1)
        batch.launch(stream=s2)
        with torch.cuda.stream(s2):
            same = torch.equal(out, want)
        torch.cuda.synchronize()
        assert same
