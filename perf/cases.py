"""The work that this library's speed is measured on: twelve listed cases and random ones of the same ranges.

Each case is a dict with a "kind" (the entry point and what surrounds it) and its sizes:

  curves    bez_eval, register evaluators: points at shared / own / uniform parameters or at in-kernel
            draws, or the fused polyline length; FP32, FP16 or BF16 control points
  texture   bez_eval through Seiler tiles read by the texture unit
  chains    bez_eval_piecewise
  spline    bez_eval_bspline / bez_eval_nurbs, clamped uniform or explicit knots
  batch     a mixed batch (Bezier, B-spline, NURBS), planned once and launched with span extraction
  surface   bez_eval_surface
  volume    bez_eval_volume
  fit       bez_mse_grad: the fused squared-error loss and its gradients
  adjoint   autograd.bezier_curve, forward and backward

Control points are U[-1, 1) (volumes: scalar fields N(0, 1)), weights U[0.5, 2), the distributions of the
benchmark's workloads.  Everything lies on the current CUDA device.
"""
import math

import numpy as np
import torch

from paper_2603_15447_gb300 import autograd, bez

STREAM = 2  # stream id of the in-kernel draws


def listed():
    return [
        # the smallest calls: a handful of curves, where the launch and the host path count
        dict(name="curves_few", kind="curves", n=100, degree=3, dim=3, n_t=64, t="shared", out="points",
             dtype="f32", variant="AUTO"),
        # outlines and strokes flattened to polylines: many short 2D cubics on one grid
        dict(name="curves_outlines", kind="curves", n=60013, degree=3, dim=2, n_t=40, t="uniform", out="points",
             dtype="f32", variant="AUTO"),
        # the benchmark's headline: 1,048,576 cubics x 1024 in-kernel draws, fused lengths
        dict(name="curves_lengths", kind="curves", n=1 << 20, degree=3, dim=3, n_t=1024, t="draws", out="length",
             dtype="f32", variant="AUTO"),
        # the same workload through the texture unit, at its 2e-3 accuracy setting
        dict(name="texture_lengths", kind="texture", n=131072, degree=3, n_t=1024, t="draws", out="length",
             spread=4, format="UNORM16"),
        # the benchmark's C0 chains of 64 quadratic segments, 65,536 draws each
        dict(name="chains_lengths", kind="chains", n=2048, segments=64, degree=2, dim=3, n_t=65536, t="draws",
             out="length", variant="AUTO"),
        # cubic B-spline curves (camera paths, profiles) sampled on one parameter list
        dict(name="spline_cubic", kind="spline", n=8191, degree=3, dim=3, n_ctrl=37, n_t=256, t="shared",
             rational=False, knots=False, out="points"),
        # quadratic NURBS with their own knot vectors and parameters, as a CAD file has them
        dict(name="spline_nurbs", kind="spline", n=4099, degree=2, dim=3, n_ctrl=20, n_t=200, t="own",
             rational=True, knots=True, out="points"),
        # the benchmark's mixed batch: 262,144 curves of every type, 16 to 4096 samples each
        dict(name="batch_mixed", kind="batch", n=262144, dim=3, max_samples=4096),
        # the benchmark's bicubic patches on 32 x 32 grids
        dict(name="surface_bicubic", kind="surface", n=65536, du=3, dv=3, dim=3, nu=32, nv=32, dtype="f32"),
        # free-form deformation: a 3D displacement lattice sampled on a voxel grid
        dict(name="volume_lattice", kind="volume", n=1000, du=3, dv=3, dw=3, dim=3, nu=20, nv=24, nw=28,
             dtype="f32"),
        # the benchmark's fitting step: 65,536 cubics, 512 samples with their own parameters
        dict(name="fit_cubic", kind="fit", n=65536, degree=3, dim=3, n_t=512, t="own", rational=False),
        # training through torch's autograd: rational quadratics (conic arcs) in the plane
        dict(name="adjoint_conics", kind="adjoint", n=10007, degree=2, dim=2, n_t=300, t="own", rational=True),
    ]


# ---------------------------------------------------------------- random cases

def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["curves", "curves", "texture", "chains", "spline", "spline", "batch", "surface", "volume",
                       "fit", "adjoint"])
    dim = rng.choice([3, 3, 3, 2, 2, 1, 4])
    if kind == "curves":
        t = rng.choice(["shared", "own", "uniform", "draws"])
        out = "length" if rng.random() < 0.3 else "points"
        n_t = _log(rng, 8, 4096)
        most = (400_000_000 if t == "draws" else 60_000_000) if out == "length" else 40_000_000
        return dict(kind=kind, n=_log(rng, 32, min(1 << 20, most // n_t)), degree=rng.choice([1, 2, 2, 3, 3, 3, 4, 5, 7]),
                    dim=dim, n_t=n_t, t=t, out=out, dtype=rng.choice(["f32", "f32", "f32", "f16", "bf16"]),
                    variant=rng.choice(["AUTO", "AUTO", "DECASTELJAU"]))
    if kind == "texture":
        out = rng.choice(["length", "points"])
        n_t = _log(rng, 32, 2048)
        most = 134_000_000 if out == "length" else 30_000_000
        return dict(kind=kind, n=_log(rng, 256, min(131072, most // n_t)), degree=rng.choice([2, 3, 3]), n_t=n_t,
                    t="draws" if out == "length" else "shared", out=out, spread=rng.choice([4, 8]),
                    format=rng.choice(["AUTO", "UNORM16"]))
    if kind == "chains":
        out = rng.choice(["length", "points"])
        n_t = _log(rng, 64, 65536)
        most = 100_000_000 if out == "length" else 30_000_000
        return dict(kind=kind, n=_log(rng, 16, min(16384, most // n_t)), segments=_log(rng, 2, 64),
                    degree=rng.choice([2, 2, 3]), dim=rng.choice([3, 3, 2]), n_t=n_t,
                    t=rng.choice(["draws", "uniform"]), out=out, variant=rng.choice(["AUTO", "HORNER_CENTRED"]))
    if kind == "spline":
        degree = rng.choice([1, 2, 3, 3, 3, 4, 5])
        n_t = _log(rng, 16, 4096)
        return dict(kind=kind, n=_log(rng, 16, min(65536, 30_000_000 // n_t)), degree=degree, dim=rng.choice([3, 3, 2]),
                    n_ctrl=rng.randint(max(4, degree + 1), 64), n_t=n_t, t=rng.choice(["shared", "own", "uniform"]),
                    rational=rng.random() < 0.5, knots=rng.random() < 0.4,
                    out="length" if rng.random() < 0.2 else "points")
    if kind == "batch":
        return dict(kind=kind, n=_log(rng, 1000, 200000), dim=rng.choice([3, 3, 2]), max_samples=_log(rng, 256, 4096))
    if kind == "surface":
        nu, nv = rng.randint(4, 96), rng.randint(4, 96)
        deg = (3, 3) if rng.random() < 0.5 else (rng.randint(1, 5), rng.randint(1, 5))
        return dict(kind=kind, n=_log(rng, 16, min(65536, 40_000_000 // (nu * nv))), du=deg[0], dv=deg[1],
                    dim=rng.choice([3, 3, 3, 4, 1]), nu=nu, nv=nv, dtype=rng.choice(["f32", "f32", "f16"]))
    if kind == "volume":
        deg = (3, 3, 3) if rng.random() < 0.5 else tuple(rng.randint(1, 3) for _ in range(3))
        nu, nv, nw = (rng.randint(4, 32) for _ in range(3))
        return dict(kind=kind, n=_log(rng, 4, min(4096, 30_000_000 // (nu * nv * nw))), du=deg[0], dv=deg[1], dw=deg[2],
                    dim=rng.choice([1, 3]), nu=nu, nv=nv, nw=nw, dtype="f32")
    n_t = _log(rng, 32, 1024)
    return dict(kind=kind, n=_log(rng, 64, min(65536, (32_000_000 if kind == "fit" else 12_000_000) // n_t)),
                degree=rng.choice([2, 3, 3, 4, 5]), dim=rng.choice([3, 3, 2]), n_t=n_t, t=rng.choice(["own", "own", "shared"]),
                rational=rng.random() < 0.35)


# ---------------------------------------------------------------- inputs

class _Gen:
    """Seeded draws on the current device."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def unit(self, *shape):
        return torch.rand(shape, generator=self.g, device="cuda")

    def uniform(self, *shape):
        return self.unit(*shape) * 2 - 1

    def weights(self, *shape):
        return self.unit(*shape) * 1.5 + 0.5

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def params(self, case, hi=1.0):
        """The parameter array of a case (None where the kernel makes the parameters), sorted along a curve."""
        if case["t"] == "shared":
            return torch.sort(self.unit(case["n_t"]) * hi).values
        if case["t"] == "own":
            return torch.sort(self.unit(case["n"], case["n_t"]) * hi, dim=1).values
        return None


DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
T_MODES = {"shared": bez.TMode.SHARED, "own": bez.TMode.PER_CURVE, "uniform": bez.TMode.UNIFORM,
           "draws": bez.TMode.HASH}
OUT_MODES = {"points": bez.OutMode.POINTS, "length": bez.OutMode.POLYLINE_LENGTH}


def _knots(g, case):
    """Clamped knot vectors over [0, 1] with uneven interior knots, one per curve."""
    n, p, nc = case["n"], case["degree"], case["n_ctrl"]
    gaps = g.unit(n, nc - p) + 0.25
    inner = (torch.cumsum(gaps, 1) / gaps.sum(1, keepdim=True))[:, :-1]
    zeros, ones = torch.zeros((n, p + 1), device="cuda"), torch.ones((n, p + 1), device="cuda")
    return torch.cat([zeros, inner, ones], 1).contiguous()


def _batch_curves(case, seed):
    """Descriptors of a mixed batch: half Bezier curves of degree 1..7, a quarter cubic B-splines, a quarter NURBS
    of degree 1..7; 4 to 64 control points and 16 to max_samples samples, uniform in their logarithm.  The curves
    are the case's, their order the seed's."""
    n, dim = case["n"], case["dim"]
    r = np.random.default_rng(n)
    kind = np.searchsorted([0.5, 0.75], r.random(n), side="right").astype(np.int32)
    degree = np.where(kind == 1, 3, r.integers(1, 8, n)).astype(np.int32)
    low = np.maximum(4, degree + 1)
    n_ctrl = np.where(kind == 0, degree + 1, low + np.floor(r.random(n) * (65 - low))).astype(np.int32)
    n_samples = np.exp(r.uniform(np.log(16), np.log(case["max_samples"] + 1), n)).astype(np.int32)
    order = np.random.default_rng(seed).permutation(n)
    kind, degree, n_ctrl, n_samples = kind[order], degree[order], n_ctrl[order], n_samples[order]

    def offsets(sizes):
        return np.concatenate([[0], np.cumsum(sizes.astype(np.int64))])

    ctrl, weight, out = offsets(n_ctrl * dim), offsets(np.where(kind == 2, n_ctrl, 0)), offsets(n_samples * dim)
    desc = bez.descriptors(kind, degree, n_ctrl, n_samples, ctrl[:-1], weight[:-1], out[:-1])
    return desc, int(ctrl[-1]), int(weight[-1]), int(out[-1])


def _batch_pools(case, seed):
    desc, n_ctrl, n_weight, n_out = _batch_curves(case, seed)
    g = _Gen(seed)
    return desc, g.uniform(n_ctrl), g.weights(max(n_weight, 1)), n_out


def _inputs(case, seed):
    """The arrays of every kind but batch."""
    g, kind = _Gen(seed), case["kind"]
    n, dim = case["n"], case.get("dim", 3)
    x = {"seed": seed}
    if kind in ("curves", "texture"):
        x["ctrl"] = g.uniform(n, case["degree"] + 1, dim).to(DTYPES[case.get("dtype", "f32")])
        x["t"] = g.params(case)
    elif kind == "chains":
        x["ctrl"], x["t"] = g.uniform(n, case["segments"] * case["degree"] + 1, dim), None
    elif kind == "spline":
        x["ctrl"], x["t"] = g.uniform(n, case["n_ctrl"], dim), g.params(case)
        x["weights"] = g.weights(n, case["n_ctrl"]) if case["rational"] else None
        x["knots"] = _knots(g, case) if case["knots"] else None
    elif kind == "surface":
        x["ctrl"] = g.uniform(n, case["du"] + 1, case["dv"] + 1, dim).to(DTYPES[case["dtype"]])
    elif kind == "volume":
        shape = (n, case["du"] + 1, case["dv"] + 1, case["dw"] + 1, dim)
        x["ctrl"] = g.normal(*shape) if dim == 1 else g.uniform(*shape)
    else:  # fit, adjoint
        x["ctrl"], x["t"] = g.uniform(n, case["degree"] + 1, dim), g.params(case)
        x["weights"] = g.weights(n, case["degree"] + 1) if case["rational"] else None
        # what arrives per sample: points near the unit cube's curves, or an upstream gradient
        x["target"] = g.uniform(n, case["n_t"], dim)
    return x


def prepare(case, seed):
    if case["kind"] == "batch":
        desc, ctrl, weights, n_out = _batch_pools(case, seed)
        out = torch.empty(n_out, device="cuda")
        return {"case": case, "out": out, "batch": bez.Batch(desc, case["dim"], ctrl, weights, out)}
    x = _inputs(case, seed)
    if case["kind"] == "adjoint":
        for k in ("ctrl", "t", "weights"):
            if x[k] is not None:
                x[k].requires_grad_()
    return dict(x, case=case)


# ---------------------------------------------------------------- one pass

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "batch":
        state["batch"].launch()
        return state["out"]
    ctrl = state["ctrl"]
    if kind == "surface":
        return bez.bez_eval_surface(ctrl, c["nu"], c["nv"])
    if kind == "volume":
        return bez.bez_eval_volume(ctrl, c["nu"], c["nv"], c["nw"])
    t = state["t"]
    if kind == "fit":
        loss, g_ctrl, g_weights, g_t = bez.bez_mse_grad(ctrl, t, state["target"], weights=state["weights"])
        return {"loss": loss, "ctrl": g_ctrl, "weights": g_weights, "t": g_t}
    if kind == "adjoint":
        wanted = [v for v in (ctrl, t, state["weights"]) if v is not None]
        points = autograd.bezier_curve(ctrl, t, state["weights"])
        return [points.detach(), *torch.autograd.grad(points, wanted, state["target"])]
    kw = dict(n_t=c["n_t"], t_mode=T_MODES[c["t"]], out_mode=OUT_MODES[c["out"]], seed=state["seed"], stream_id=STREAM)
    if kind == "curves":
        return bez.bez_eval(ctrl, t, variant=bez.Variant[c["variant"]], **kw)
    if kind == "texture":
        return bez.bez_eval(ctrl, t, variant=bez.Variant.TEX_SEILER, tex_spread=c["spread"],
                            tex_format=bez.TexFormat[c["format"]], **kw)
    if kind == "chains":
        return bez.bez_eval_piecewise(ctrl, c["segments"], c["degree"], t, variant=bez.Variant[c["variant"]], **kw)
    if c["rational"]:
        return bez.bez_eval_nurbs(ctrl, state["weights"], c["degree"], t, knots=state["knots"], **kw)
    return bez.bez_eval_bspline(ctrl, c["degree"], t, knots=state["knots"], **kw)


# ---------------------------------------------------------------- the least work of a pass

def work(case):
    c, kind = case, case["kind"]
    n, dim = c["n"], c.get("dim", 3)
    if kind == "batch":
        # means over the draws of _batch_curves
        samples = n * (c["max_samples"] - 16) / math.log(c["max_samples"] / 16)
        ctrl = n * (0.5 * 5 + 0.25 * 34 + 0.25 * 36)
        weights = n * 0.25 * 36
        return {"bytes": 4 * (samples * dim + ctrl * dim + weights), "flops": samples * dim * 2 * 3.75}
    if kind == "surface":
        pts = n * c["nu"] * c["nv"]
        size = 4 if c["dtype"] == "f32" else 2
        ctrl = n * (c["du"] + 1) * (c["dv"] + 1) * dim
        return {"bytes": 4 * pts * dim + size * ctrl, "flops": 2 * dim * (pts * (c["dv"] + 1) + n * c["nu"] * (c["du"] + 1) * (c["dv"] + 1))}
    if kind == "volume":
        pts = n * c["nu"] * c["nv"] * c["nw"]
        ctrl = n * (c["du"] + 1) * (c["dv"] + 1) * (c["dw"] + 1) * dim
        return {"bytes": 4 * (pts * dim + ctrl), "flops": 2 * dim * (pts * (c["dw"] + 1) + n * c["nu"] * c["nv"] * (c["dv"] + 1) * (c["dw"] + 1))}
    pts = n * c["n_t"]
    t_bytes = 4 * (pts if c["t"] == "own" else c["n_t"] if c["t"] == "shared" else 0)
    if kind in ("fit", "adjoint"):
        ctrl = n * (c["degree"] + 1) * (dim + (1 if c["rational"] else 0))
        # fit reads t and the targets and writes dt; adjoint also writes the points on its way
        passes = dim + (dim if kind == "adjoint" else 0)
        return {"bytes": 2 * t_bytes + 4 * (pts * passes + 2 * ctrl),
                "flops": pts * dim * (6 * c["degree"] + 8)}
    size = 4 if c.get("dtype", "f32") == "f32" else 2
    per = c["segments"] * c["degree"] + 1 if kind == "chains" else c["n_ctrl"] if kind == "spline" else c["degree"] + 1
    in_bytes = size * n * per * dim
    if kind == "spline":
        in_bytes += 4 * n * ((per if c["rational"] else 0) + (per + c["degree"] + 1 if c["knots"] else 0))
    length = c["out"] == "length"
    flops = pts * (2 * c["degree"] * dim + (3 * dim + 2 if length else 0))
    return {"bytes": in_bytes + t_bytes + 4 * (n if length else pts * dim), "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits

M32 = 0xFFFFFFFF


def _mix(x):
    """lowbias32 on 32-bit values held in int64 tensors or Python ints."""
    x = x ^ (x >> 16)
    x = (x * 0x7FEB352D) & M32
    x = x ^ (x >> 15)
    x = (x * 0x846CA68B) & M32
    return x ^ (x >> 16)


def _draws(seed, c0, c1, n_t):
    """The in-kernel draws of curves c0..c1: 23-bit uniforms in [0, 1), exact."""
    key = _mix((seed & M32) ^ _mix((seed >> 32) ^ _mix(STREAM)))
    c = torch.arange(c0, c1, device="cuda", dtype=torch.int64)
    j = torch.arange(n_t, device="cuda", dtype=torch.int64)
    return (_mix(_mix(c ^ key)[:, None] ^ j[None, :]) >> 9).double() * 2.0 ** -23


def _grid(n):
    """fl32(j) / fl32(n - 1), as FP32 values."""
    j = torch.arange(n, device="cuda", dtype=torch.float32)
    return (j / max(n - 1, 1)).double()


def _exact_t(case, x, c0, c1, scale=1):
    """FP64 copies of the FP32 parameters of curves c0..c1: [n_t] or [c1 - c0][n_t]."""
    if case["t"] == "shared":
        return x["t"].double()
    if case["t"] == "own":
        return x["t"][c0:c1].double()
    u = _grid(case["n_t"]) if case["t"] == "uniform" else _draws(x["seed"], c0, c1, case["n_t"])
    return (u.float() * scale).double() if scale != 1 else u


def _bernstein(t, d):
    """[..., d + 1] Bernstein values."""
    i = torch.arange(d + 1, device="cuda")
    binom = torch.tensor([math.comb(d, k) for k in range(d + 1)], device="cuda", dtype=torch.float64)
    return binom * t[..., None] ** i * (1 - t[..., None]) ** (d - i)


def _bezier(b, t):
    """Curves b [n][d + 1][dim] at t [n_t] or [n][n_t]."""
    B = _bernstein(t, b.shape[1] - 1)
    return torch.einsum("ji,nik->njk" if t.ndim == 1 else "nji,nik->njk", B, b)


def _length(p):
    return (p[:, 1:] - p[:, :-1]).norm(dim=-1).sum(1)


def _de_boor(h, U, t, p):
    """Splines with homogeneous or plain points h [n][n_ctrl][k], knots U [n][n_ctrl + p + 1], t [n][n_t]."""
    n, nc, k = h.shape
    s = (torch.searchsorted(U[:, p:nc].contiguous(), t.contiguous(), right=True) - 1).clamp(0, nc - p - 1) + p
    at = s[..., None] - p + torch.arange(p + 1, device="cuda")
    row = torch.arange(n, device="cuda")[:, None, None]
    d = h[row, at]                                                           # [n][n_t][p + 1][k]
    for r in range(1, p + 1):
        j = torch.arange(r, p + 1, device="cuda")
        lo = torch.gather(U, 1, (s[..., None] - p + j).flatten(1)).view(n, -1, p + 1 - r)
        hi = torch.gather(U, 1, (s[..., None] + 1 + j - r).flatten(1)).view(n, -1, p + 1 - r)
        a = ((t[..., None] - lo) / (hi - lo))[..., None]
        d = (1 - a) * d[:, :, :-1] + a * d[:, :, 1:]
    return d[:, :, 0]


def _uniform_knots(nc, p):
    inner = torch.arange(1, nc - p, device="cuda", dtype=torch.float64) / (nc - p)
    return torch.cat([torch.zeros(p + 1, device="cuda", dtype=torch.float64), inner,
                      torch.ones(p + 1, device="cuda", dtype=torch.float64)])


def _splines(ctrl, weights, U, t, p):
    if weights is None:
        return _de_boor(ctrl.double(), U, t, p)
    w = weights.double()[..., None]
    h = _de_boor(torch.cat([ctrl.double() * w, w], 2), U, t, p)
    return h[..., :-1] / h[..., -1:]


def _exact_batch(case, seed):
    desc, ctrl, weights, n_out = _batch_pools(case, seed)
    dim = case["dim"]
    out = torch.empty(n_out, device="cuda", dtype=torch.float64)
    # one group per control-point count and degree: a Bezier curve is the spline with degree + 1 of them
    group = desc["type"].astype(np.int64) * 10000 + desc["degree"] * 1000 + desc["n_ctrl"]
    order = np.argsort(group, kind="stable")
    for ids in np.split(order, np.nonzero(np.diff(group[order]))[0] + 1):
        kind, p, nc = (int(desc[f][ids[0]]) for f in ("type", "degree", "n_ctrl"))
        while len(ids):
            m = max(1, int(np.searchsorted(np.cumsum(desc["n_samples"][ids]), 4_000_000)))
            part, ids = ids[:m], ids[m:]
            d = {f: torch.from_numpy(desc[f][part].astype(np.int64)).cuda() for f in ("n_samples", "ctrl_off", "weight_off", "out_off")}
            # one row per curve, cut to the samples it has
            n_s, most = d["n_samples"], int(desc["n_samples"][part].max())
            rows = max(1, 8_000_000 // most)
            for r0 in range(0, m, rows):
                r = slice(r0, min(r0 + rows, m))
                j = torch.arange(most, device="cuda")
                t = (j.float()[None, :] / (n_s[r, None] - 1).clamp(min=1).float()).clamp(max=1).double()
                b = ctrl[(d["ctrl_off"][r, None] + torch.arange(nc * dim, device="cuda"))].view(-1, nc, dim)
                w = weights[d["weight_off"][r, None] + torch.arange(nc, device="cuda")] if kind == 2 else None
                U = _uniform_knots(nc, p).expand(len(b), -1).contiguous()
                pts = _splines(b, w, U, t, p) if kind else _bezier(b.double(), t)
                live = j[None, :] < n_s[r, None]
                at = d["out_off"][r, None] + j[None, :] * dim
                out[(at[live][:, None] + torch.arange(dim, device="cuda"))] = pts[live]
    return out


def _exact_gradients(case, x):
    """Per-curve loss (fit) or points (adjoint), and the gradients, by torch's autograd in FP64."""
    n, fit = case["n"], case["kind"] == "fit"
    parts, g_shared = [], 0
    step = max(1, 4_000_000 // case["n_t"])
    for c0 in range(0, n, step):
        s = slice(c0, min(c0 + step, n))
        ctrl = x["ctrl"].detach()[s].double().requires_grad_()
        t = (x["t"].detach() if case["t"] == "shared" else x["t"].detach()[s]).double().requires_grad_()
        w = x["weights"].detach()[s].double().requires_grad_() if case["rational"] else None
        target = x["target"][s].double()
        if w is None:
            pts = _bezier(ctrl, t)
        else:
            h = _bezier(torch.cat([ctrl * w[..., None], w[..., None]], 2), t)
            pts = h[..., :-1] / h[..., -1:]
        wanted = [v for v in (ctrl, t, w) if v is not None]
        if fit:
            first = ((pts - target) ** 2).sum((1, 2)) / (n * case["n_t"] * case["dim"])
            got = torch.autograd.grad(first.sum(), wanted)
        else:
            first = pts
            got = torch.autograd.grad(pts, wanted, target)
        if case["t"] == "shared":
            g_shared = g_shared + got[1]
        parts.append([first.detach(), *got])
    whole = [torch.cat(v) for v in zip(*parts)]
    if case["t"] == "shared":
        whole[2] = g_shared
    if not fit:
        return whole
    return {"loss": whole[0], "ctrl": whole[1], "t": whole[2], "weights": whole[3] if case["rational"] else None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    x = _inputs(case, seed)
    if kind in ("fit", "adjoint"):
        return _exact_gradients(case, x)
    if kind == "surface":
        Bu, Bv = _bernstein(_grid(case["nu"]), case["du"]), _bernstein(_grid(case["nv"]), case["dv"])
        return torch.einsum("nijk,ai,bj->nabk", x["ctrl"].double(), Bu, Bv)
    if kind == "volume":
        B = [_bernstein(_grid(case[g]), case[d]) for g, d in (("nu", "du"), ("nv", "dv"), ("nw", "dw"))]
        return torch.einsum("nijlk,ai,bj,cl->nabck", x["ctrl"].double(), *B)
    n, n_t, parts = case["n"], case["n_t"], []
    step = max(1, 8_000_000 // n_t)
    for c0 in range(0, n, step):
        c1 = min(c0 + step, n)
        ctrl = x["ctrl"][c0:c1].double()
        if kind in ("curves", "texture"):
            p = _bezier(ctrl, _exact_t(case, x, c0, c1))
        elif kind == "chains":
            t = _exact_t(case, x, c0, c1, case["segments"]).expand(c1 - c0, -1)
            k = t.floor().long().clamp(0, case["segments"] - 1)
            B = _bernstein(t - k, case["degree"])
            row = torch.arange(c1 - c0, device="cuda")[:, None]
            p = sum(B[..., i, None] * ctrl[row, k * case["degree"] + i] for i in range(case["degree"] + 1))
        else:
            U = (x["knots"][c0:c1].double() if case["knots"]
                 else _uniform_knots(case["n_ctrl"], case["degree"]).expand(c1 - c0, -1).contiguous())
            w = x["weights"][c0:c1] if case["rational"] else None
            p = _splines(ctrl, w, U, _exact_t(case, x, c0, c1).expand(c1 - c0, -1), case["degree"])
        parts.append(_length(p) if case["out"] == "length" else p)
    return torch.cat(parts)
