"""GPU parity of 2D batches (fixed-degree kernels) at sample counts around the
runs and tiles of a warp, every degree and curve type, both representations,
against the FP64 oracle at 1e-6 of the control polygon's diagonal (unit-square
points, so the floor 2^-4 of the secondary normaliser is never reached)."""
import numpy as np
import pytest

import oracle
from gpu_util import need_gpu, normalised_error_ctrl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("repr", [0, 1])
def test_runs_and_tiles(repr):
    torch = need_gpu()
    from paper_2603_15447_gb300 import bez
    rng = np.random.default_rng(11 + repr)
    rows, ctrl, wts, want = [], [], [], []
    off = [0, 0, 0]
    for kind in (0, 1, 2):
        for p in range(1, 8):
            for n_s in (1, 31, 33, 64, 65, 128, 129, 256, 257, 600):
                n_c = p + 1 if kind == 0 else p + 1 + int(rng.integers(0, 9))
                # a polygon with two opposite corners of the square: its diagonal is at least 1
                b = rng.uniform(0, 1, (1, n_c, 2)).astype(np.float32)
                b[0, 0], b[0, -1] = 0.0, 1.0
                w = rng.uniform(0.5, 2, (1, n_c)).astype(np.float32)
                rows.append((kind, p, n_c, n_s, *off))
                t = oracle.grid(n_s)
                if kind == 0:
                    ref = oracle.bezier(b, t)
                else:
                    ref = oracle.bspline(b, p, t, weights=w if kind == 2 else None)
                want.append((off[2], n_s, b, ref))
                ctrl.append(b.ravel())
                off[0] += 2 * n_c
                if kind == 2:
                    wts.append(w.ravel())
                    off[1] += n_c
                off[2] += 2 * n_s
    out = torch.full((off[2],), float("nan"), device="cuda")
    desc = bez.descriptors(*[np.array(c) for c in zip(*rows)])
    bez.Batch(desc, 2, torch.from_numpy(np.concatenate(ctrl)).cuda(), torch.from_numpy(np.concatenate(wts)).cuda(),
              out, repr=repr).launch()
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for o, n_s, b, ref in want:
        assert normalised_error_ctrl(got[o:o + 2 * n_s].reshape(1, n_s, 2), ref, b).max() <= 1e-6
