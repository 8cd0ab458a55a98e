"""The launch shape a batch plan takes by default, by its samples, and its
results under it against the static schedule at 512 samples an item."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("samples, graph, chunk, schedule", [
    (1_000_000, True, 256, 0), (4_000_000, True, 512, 0), (39_000_000, False, 512, 0), (61_000_000, True, 1024, 0),
    (99_000_000, True, 1024, 0), (100_000_000, True, 2048, 0), (161_000_000, True, 1024, 1),
    (161_000_000, False, 2048, 0)])
def test_default_shape(samples, graph, chunk, schedule):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    n, dim = 1000, 2
    n_s, i = samples // n, np.arange(n)
    rng = np.random.default_rng(1)
    desc = bez.descriptors(np.zeros(n), np.full(n, 3), np.full(n, 4), np.full(n, n_s), i * 8, i * 0, i * n_s * dim)
    ctrl = torch.from_numpy(rng.uniform(-1, 1, n * 8).astype(np.float32)).cuda()
    out, ref = (torch.full((n * n_s * dim,), float("nan"), device="cuda") for _ in range(2))
    batch = bez.Batch(desc, dim, ctrl, None, out, use_graph=graph)
    got = batch.config()
    assert (got["chunk"], got["schedule"], got["threads"]) == (chunk, schedule, 128)
    batch.launch()
    bez.Batch(desc, dim, ctrl, None, ref, chunk=512, schedule=0).launch()
    assert torch.equal(out, ref)                       # a sample's value does not depend on its item
