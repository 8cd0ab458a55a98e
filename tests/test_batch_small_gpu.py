"""The two paths of 2D batches: the fixed-degree class kernels at sizes where a
plan takes the generic kernel by default, and the step between them."""
import functools

import numpy as np
import pytest

import oracle
import test_batch_2d_gpu
from gpu_util import need_gpu, normalised_error_ctrl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("repr", [0, 1])
def test_class_kernels(repr, monkeypatch):
    need_gpu()
    from paper_2603_15447_gb300 import bez
    monkeypatch.setattr(bez, "Batch", functools.partial(bez.Batch, chunk=512))  # an item size of their own
    test_batch_2d_gpu.test_runs_and_tiles(repr)


@pytest.mark.parametrize("n, launches", [(3999, 2), (4000, 4)])
def test_step(n, launches):
    # one curve of 257 samples (two items) among n - 1 of 16; two degrees
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(n)
    n_s = np.full(n, 16)
    n_s[7] = 257
    degree = np.where(np.arange(n) < n // 2, 2, 3)
    ctrl = rng.uniform(0, 1, (n, 4, 2)).astype(np.float32)
    ctrl[:, 0], ctrl[:, 2:] = 0.0, 1.0                 # diagonal >= 1
    off = np.concatenate([[0], np.cumsum(n_s)]) * 2
    desc = bez.descriptors(np.zeros(n), degree, degree + 1, n_s, np.arange(n) * 8, np.zeros(n), off[:-1])
    out = torch.full((int(off[-1]),), float("nan"), device="cuda")
    ctx = bez.Context(0)
    batch = bez.Batch(desc, 2, torch.from_numpy(ctrl.ravel()).cuda(), None, out, ctx=ctx)
    ctx.reset_stats()
    batch.launch()
    assert ctx.stats()["launches"] == launches          # an extraction and an evaluation per class
    got = out.cpu().numpy()
    for c in (0, 7, n // 2 - 1, n // 2, n - 1):
        b = ctrl[c:c + 1, :degree[c] + 1]
        ref = oracle.bezier(b, oracle.grid(n_s[c]))
        assert normalised_error_ctrl(got[off[c]:off[c + 1]].reshape(1, -1, 2), ref, b).max() <= 1e-6
    assert np.isfinite(got).all()


def test_tuned_shapes_are_kept_apart(tmp_path, monkeypatch):
    """A shape tuned for the class kernels is not taken for a plan of one generic kernel, nor the other way round."""
    torch = need_gpu()
    import json
    from paper_2603_15447_gb300 import bez
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("BEZ_AUTOTUNE_CACHE", str(cache))
    n, n_s, dim = 500, 64, 2
    i = np.arange(n)
    desc = bez.descriptors(np.zeros(n), np.full(n, 2), np.full(n, 3), np.full(n, n_s), i * 3 * dim, i * 0, i * n_s * dim)
    ctrl, out = torch.rand(n * 3 * dim, device="cuda"), torch.empty(n * n_s * dim, device="cuda")
    for chunk in (0, 512):
        bez.Batch(desc, dim, ctrl, None, out, autotune=True, chunk=chunk)
    keys = {k for k in json.loads(cache.read_text()) if k.startswith("batch-v3:setup1:n9:dim2")}
    assert {k.endswith(":one") for k in keys} == {True, False}
