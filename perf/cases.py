"""The work that users of the library have it do, as timed cases.

Each case is one call (or one short sequence of calls) of the public entry points, over the sizes of the
repository's workloads: the operators A and A^T on parallel, cone, helical and explicit rays, with the exact and the
learned footprint, the gradient of a training batch of the learned footprint, and a short CGLS reconstruction.

Outputs are the whole projections, coefficient arrays and gradients.  `exact` evaluates the same operators in FP64
with plain torch: every line is cut at the knot planes of the three axes and each polynomial piece of the spline is
integrated by Gauss-Legendre nodes, which shares nothing with the library's march.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_11078_gb300 import inputs as I
from paper_2511_11078_gb300 import recon, spl

# FP64 gathers of one operator that `exact` does at most (about 10 s on the GPU)
EXACT_LIMIT = 1.0e11


# ---------------------------------------------------------------- the cases
def listed():
    """What each stands for:

    small-gradient     the oracle-sized workload: one gradient of the least-squares loss through autograd, where
                       launches and the latency of a single ray count
    rays-gradient      explicit rays on an odd grid (no view structure), the same gradient
    tilt-cubic         a single-axis tilt series plus random directions, 128^3, the autograd workload
    tilt-linear        the same with linear splines
    cone-forward       A of the 256^3 circular cone workload (every third of its 360 views)
    cone-adjoint       its A^T
    helical-forward    A of the 512^3 helical workload (36 of its 720 views), the largest grid
    helical-adjoint    its A^T
    learned-forward    A with the learned footprint on the 256^3 cone workload (6 views)
    learned-adjoint    its A^T
    learned-gradient   gradient of the footprint network on a training batch of 8192 samples
    cgls-quadratic     two CGLS iterations of the head-sized quadratic reconstruction (180 x 180 x 50, 200 cone views)
    """
    return [
        dict(name="small-gradient", op="gradient", kind="parallel", degree=3, nx=24, ny=24, nz=24, views=32, tilt=0,
             nu=32, nv=32, pitch=1.0),
        dict(name="rays-gradient", op="gradient", kind="rays", degree=3, nx=99, ny=90, nz=77, rays=150001),
        dict(name="tilt-cubic", op="gradient", kind="parallel", degree=3, nx=128, ny=128, nz=128, views=64, tilt=180,
             nu=192, nv=192, pitch=1.0),
        dict(name="tilt-linear", op="gradient", kind="parallel", degree=1, nx=128, ny=128, nz=128, views=64, tilt=180,
             nu=192, nv=192, pitch=1.0),
        dict(name="cone-forward", op="forward", kind="cone", degree=3, nx=256, ny=256, nz=256, views=120, nu=384,
             nv=384, pitch=1.2, sod=1000.0, sdd=1500.0, turns=1.0),
        dict(name="cone-adjoint", op="adjoint", kind="cone", degree=3, nx=256, ny=256, nz=256, views=120, nu=384,
             nv=384, pitch=1.2, sod=1000.0, sdd=1500.0, turns=1.0),
        dict(name="helical-forward", op="forward", kind="cone", degree=3, nx=512, ny=512, nz=512, views=36, nu=768,
             nv=768, pitch=0.8, sod=1000.0, sdd=1500.0, turns=2.0),
        dict(name="helical-adjoint", op="adjoint", kind="cone", degree=3, nx=512, ny=512, nz=512, views=36, nu=768,
             nv=768, pitch=0.8, sod=1000.0, sdd=1500.0, turns=2.0),
        dict(name="learned-forward", op="learned-forward", kind="cone", degree=3, nx=256, ny=256, nz=256, views=6,
             nu=384, nv=384, pitch=1.2, sod=1000.0, sdd=1500.0, turns=1.0),
        dict(name="learned-adjoint", op="learned-adjoint", kind="cone", degree=3, nx=256, ny=256, nz=256, views=6,
             nu=384, nv=384, pitch=1.2, sod=1000.0, sdd=1500.0, turns=1.0),
        dict(name="learned-gradient", op="learned-gradient", kind="batch", degree=3, batch=8192),
        dict(name="cgls-quadratic", op="cgls", kind="cone", degree=2, nx=180, ny=180, nz=50, views=200, nu=180, nv=50,
             pitch=2.2, sod=720.0, sdd=1440.0, turns=1.0, iters=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: grids of 20 to 400 per axis with odd sizes and unequal axes, detectors that
    cover them, 1 to 200 views, all the kinds and operations of the list."""
    op = rng.choice(["gradient", "gradient", "gradient", "forward", "adjoint", "forward", "adjoint", "cgls",
                     "learned-forward", "learned-adjoint", "learned-gradient"])
    if op == "learned-gradient":
        return dict(op=op, kind="batch", degree=3, batch=_log_int(rng, 500, 16384))
    degree = 3 if op.startswith("learned") else rng.choice([3, 3, 3, 2, 1])
    n = _log_int(rng, 20, 96 if op.startswith("learned") else 400)
    dims = [max(12, int(n * rng.uniform(0.6, 1.0))) for _ in range(3)]
    dims[rng.randrange(3)] = n
    case = dict(op=op, degree=degree, nx=dims[0], ny=dims[1], nz=dims[2])
    # rays of the pass: bounded so that no drawn case costs more than the largest listed one
    budget = (1.0e8 if op.startswith("learned") else 6.0e9) / n
    if op in ("gradient", "cgls"):
        budget /= 4.0
    kind = "cone" if op.startswith("learned") or op == "cgls" else rng.choice(["parallel", "cone", "cone", "rays"])
    case["kind"] = kind
    if kind == "rays":
        case["rays"] = max(1000, min(_log_int(rng, 5000, 600000), int(budget)))
        return case
    det = max(16, int(n * rng.uniform(1.0, 1.5)))
    case["nu"], case["nv"] = det, max(16, int(det * rng.uniform(0.6, 1.0)))
    most = max(1, min(200, int(budget / (case["nu"] * case["nv"]))))
    views = min(most, _log_int(rng, 1, 200))
    if kind == "parallel":
        tilt = rng.choice([0, views // 2])
        case.update(views=views - tilt, tilt=tilt, pitch=rng.choice([1.0, 1.0, 0.7]))
    else:
        sod = n * rng.uniform(2.0, 4.0)
        mag = rng.uniform(1.3, 2.0)
        case.update(views=views, pitch=round(mag * rng.uniform(0.6, 1.2), 3), sod=round(sod, 2),
                    sdd=round(sod * mag, 2), turns=rng.choice([1.0, 1.0, 2.0]))
    if op == "cgls":
        case["iters"] = 2
    return case


# ---------------------------------------------------------------- inputs
def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _geometry(case, seed):
    """Pose arrays: fixed by the case, except explicit rays and random directions, which the seed draws."""
    rng = np.random.default_rng(1000 + seed)
    if case["kind"] == "rays":
        w = I.random_directions(rng, case["rays"])
        # points spread over the volume: every line crosses it
        half = 0.5 * (np.asarray(_dims(case), dtype=np.float64) - 1.0)
        s = rng.uniform(-0.8, 0.8, size=w.shape) * half + rng.uniform(-50.0, 50.0, size=(w.shape[0], 1)) * w
        return I.RayGeometry(w, s)
    if case["kind"] == "parallel":
        parts = []
        if case["tilt"]:
            parts.append(I.tilt_series(case["tilt"], case["nu"], case["nv"], case["pitch"]))
        if case["views"]:
            parts.append(I.parallel_views(I.random_directions(rng, case["views"]), case["nu"], case["nv"],
                                          case["pitch"]))
        cat = [np.concatenate([getattr(p, f) for p in parts]) for f in ("src", "det_center", "det_u", "det_v")]
        return I.ViewGeometry("parallel", *cat, case["nu"], case["nv"])
    feed = 0.0 if case["turns"] == 1.0 else 0.5 * case["nv"] * case["pitch"] * case["sod"] / case["sdd"]
    return I.helical_cone(case["views"], case["sod"], case["sdd"], case["nu"], case["nv"], case["pitch"],
                          turns=case["turns"], table_feed=feed)


def _generator(seed, stream):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * (seed + 1) + stream)
    return gen


def _coefficients(case, seed):
    """An ellipsoid phantom (densities 0.2 .. 1, piecewise constant) with a weak noise texture, float32 [z][y][x]."""
    rng = np.random.default_rng(2000 + seed)
    nx, ny, nz = _dims(case)
    dims = np.array([nx, ny, nz], dtype=np.float64)
    c = torch.randn((nz, ny, nx), generator=_generator(seed, 1), device="cuda").mul_(0.02)
    axes = [torch.arange(n, device="cuda", dtype=torch.float32) - 0.5 * (n - 1) for n in (nx, ny, nz)]
    X, Y, Z = axes[0][None, None, :], axes[1][None, :, None], axes[2][:, None, None]
    for R in I.random_rotations(rng, 6):
        ctr = rng.uniform(-0.3, 0.3, 3) * dims
        semi = rng.uniform(0.08, 0.35, 3) * float(dims.min())
        q = torch.zeros((), device="cuda")
        for e in range(3):
            q = q + ((R[0, e] * (X - ctr[0]) + R[1, e] * (Y - ctr[1]) + R[2, e] * (Z - ctr[2])) / semi[e]).square()
        c += float(rng.uniform(0.2, 1.0)) * (q <= 1.0)
    return c


def _projection(shape, seed):
    """Data or a residual: mixed signs, as the adjoint meets it in an iteration."""
    return torch.randn(shape, generator=_generator(seed, 2), device="cuda")


def _network(seed):
    """Master parameters of the footprint network, uniform in +-1/sqrt(fan in), and a batch of (features, labels)."""
    rng = np.random.default_rng(3000 + seed)
    parts = []
    for fan_in, fan_out in ((5, 64), (64, 64), (64, 64), (64, 1)):
        b = 1.0 / math.sqrt(fan_in)
        parts += [rng.uniform(-b, b, fan_in * fan_out), rng.uniform(-b, b, fan_out)]
    return np.concatenate(parts).astype(np.float32)


def _batch(case, seed):
    """Training samples: directions of the chamber 0 <= w1 <= w2 <= w3, offsets in the scaled disc of radius 3, and
    labels shaped like a footprint (a bump of height about 0.45)."""
    gen = _generator(seed, 3)
    w = torch.randn((case["batch"], 3), generator=gen, device="cuda")
    w = (w / w.norm(dim=1, keepdim=True)).abs().sort(dim=1).values
    r = 3.0 * torch.rand(case["batch"], generator=gen, device="cuda").sqrt()
    a = 2.0 * math.pi * torch.rand(case["batch"], generator=gen, device="cuda")
    feat = torch.cat([w, (r * a.cos())[:, None], (r * a.sin())[:, None]], dim=1).contiguous()
    return feat, (0.45 * torch.exp(-1.5 * r * r)).contiguous()


def prepare(case, seed):
    op = case["op"]
    if op == "learned-gradient":
        mlp = spl.Mlp(case["degree"], max_batch=case["batch"], seed=1)
        mlp.set_params(_network(seed))
        feat, label = _batch(case, seed)
        return dict(op=op, mlp=mlp, feat=feat, label=label)
    geom = spl.Geometry(_dims(case), I.centred_origin(_dims(case)), _geometry(case, seed))
    mlp = None
    if op.startswith("learned"):
        mlp = spl.Mlp(case["degree"], max_batch=1024, seed=1)
        mlp.set_params(_network(seed))
    proj = recon.Projector(geom, case["degree"], spl.SPL_FP_MLP if mlp else spl.SPL_FP_QUAD, mlp)
    spl.prepare(geom, proj.basis)
    state = dict(op=op, proj=proj)
    if op in ("gradient", "forward", "learned-forward"):
        state["c"] = _coefficients(case, seed)
    if op in ("gradient", "adjoint", "learned-adjoint", "cgls"):
        state["y"] = _projection(geom.shape, seed)
    if op == "cgls":
        state["iters"] = case["iters"]
    return state


# ---------------------------------------------------------------- one pass
def run(state):
    op = state["op"]
    if op in ("forward", "learned-forward"):
        return state["proj"].forward(state["c"])
    if op in ("adjoint", "learned-adjoint"):
        return state["proj"].adjoint(state["y"])
    if op == "gradient":
        # gradient of 1/2 |A c - y|^2: the forward, the residual, the backward
        c = state["c"].detach().requires_grad_()
        p = recon.project(c, state["proj"])
        (g,) = torch.autograd.grad(p, c, p.detach() - state["y"])
        return p.detach(), g
    if op == "cgls":
        return recon.cgls(state["proj"], state["y"], state["iters"])
    grad = torch.empty(spl.MLP_PARAMS, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    state["mlp"].grad(state["feat"], state["label"], grad, loss)
    return grad, loss


# ---------------------------------------------------------------- what a pass cannot do without
def _sample_lines(case):
    """A thinned set of the case's lines (s, w) and how many lines each stands for."""
    g = _geometry(case, 0)
    if case["kind"] == "rays":
        return g.s, g.omega, 1.0
    k = np.arange(0, g.n_views, max(1, g.n_views // 24))
    iu = np.arange(0, case["nu"], max(1, case["nu"] // 24)) - 0.5 * (case["nu"] - 1)
    iv = np.arange(0, case["nv"], max(1, case["nv"] // 24)) - 0.5 * (case["nv"] - 1)
    q = (g.det_center[k, None, None] + iu[None, None, :, None] * g.det_u[k, None, None] +
         iv[None, :, None, None] * g.det_v[k, None, None]).reshape(-1, 3)
    src = np.repeat(g.src[k], iu.size * iv.size, axis=0)
    w = src if g.kind == "parallel" else q - src
    w = w / np.linalg.norm(w, axis=1, keepdims=True)
    return q, w, g.n_rays / q.shape[0]


def _crossings(case):
    """Of one operator, from the chords of the sampled lines: unit-cell pieces, (ray, basis) pairs, and the pairs in
    the plane of the lines that run parallel to a grid plane (single-axis tilt), which the pieces leave out."""
    s, w, each = _sample_lines(case)
    half = 0.5 * np.asarray(_dims(case), dtype=np.float64)
    # the knot planes bound the grid's supports: the box of half width (n + degree) / 2
    out = half + 0.5 * case["degree"]
    with np.errstate(divide="ignore", invalid="ignore"):
        t = np.stack([(-out - s) / w, (out - s) / w])
    lo, hi = np.nanmax(t.min(axis=0), axis=1), np.nanmin(t.max(axis=0), axis=1)
    chord = np.maximum(hi - lo, 0.0)
    steps = np.abs(w).sum(axis=1)
    flat = (w == 0.0).any(axis=1)
    pieces = float((chord * steps)[~flat].sum() * each)
    # a line of length L in the grid meets L (n+1)^2 sum |w_e| supports, L (n+1) sum |w_e| in its plane
    inner = chord * np.prod(half) / np.prod(out)
    m = case["degree"] + 1
    return pieces, float((inner * steps).sum() * each * m ** 2), float((inner * steps)[flat].sum() * each * m)


def work(case):
    if case["op"] == "learned-gradient":
        n = case["batch"]
        # forward, the products with the transposed weights, the weight gradients
        return {"bytes": 4.0 * (6 * n + 2 * spl.MLP_PARAMS + 1), "flops": 6.0 * 8576 * n}
    n = case["degree"]
    pieces, pairs, plane = _crossings(case)
    nc = case["nx"] * case["ny"] * case["nz"]
    nr = case["rays"] if case["kind"] == "rays" else (case["views"] + case.get("tilt", 0)) * case["nu"] * case["nv"]
    calls = {"gradient": 2, "cgls": 1 + 2 * case.get("iters", 0)}.get(case["op"], 1)
    if case["op"].startswith("learned"):
        flops = 17152.0 * pairs
    else:
        # a piece of the line: ceil((3n+1)/2) nodes, each a contraction with the (n+1)^3 live coefficients; a line
        # in a grid plane: one multiply-add per pair in the plane (the third factor is constant along it)
        m = n + 1
        flops = (pieces * ((3 * n + 2) // 2) * 2.0 * (m ** 3 + m ** 2 + m) + 2.0 * plane) * calls
    # the gradient reads c and the data and writes the projection and the gradient; the others one array of each
    moved = {"gradient": 2.0 * (nc + nr)}.get(case["op"], float(nc + nr))
    return {"bytes": 4.0 * moved, "flops": flops}


# ---------------------------------------------------------------- FP64 values
class _Exact:
    """A and A^T in FP64 for the lines of a case: pieces between knot planes, Gauss-Legendre nodes."""

    def __init__(self, case, seed):
        self.n, self.dims = case["degree"], _dims(case)
        g = _geometry(case, seed)
        if case["kind"] == "rays":
            s, w = torch.tensor(g.s, device="cuda"), torch.tensor(g.omega, device="cuda")
            self.shape = (case["rays"],)
        else:
            d = {f: torch.tensor(getattr(g, f), device="cuda") for f in ("src", "det_center", "det_u", "det_v")}
            iu = torch.arange(g.nu, device="cuda", dtype=torch.float64) - 0.5 * (g.nu - 1)
            iv = torch.arange(g.nv, device="cuda", dtype=torch.float64) - 0.5 * (g.nv - 1)
            q = (d["det_center"][:, None, None] + iu[None, None, :, None] * d["det_u"][:, None, None] +
                 iv[None, :, None, None] * d["det_v"][:, None, None])
            src = d["src"][:, None, None].expand_as(q)
            s, w = q.reshape(-1, 3), (src if g.kind == "parallel" else q - src).reshape(-1, 3)
            self.shape = (g.n_views, g.nv, g.nu)
        self.s, self.w = s, w / w.norm(dim=1, keepdim=True)
        x, wt = np.polynomial.legendre.leggauss((3 * self.n + 2) // 2)
        self.x, self.wt = x.tolist(), wt.tolist()
        # index coordinates: coefficient k at k
        self.s = self.s + torch.tensor([0.5 * (n - 1) for n in self.dims], device="cuda", dtype=torch.float64)
        knots = sum(n + self.n + 1 for n in self.dims)
        self.knots = knots
        self.gathers = float(self.s.shape[0]) * knots * len(self.x) * (self.n + 1) ** 3
        self.chunk = max(1, int(2.0e7 / knots))

    @staticmethod
    def _weights(n, g):
        """beta^n of the n+1 bases that hold a point at fraction g of their common cell."""
        t = 1.0 - g
        if n == 1:
            return [t, g]
        if n == 2:
            return [0.5 * t * t, 0.5 + g * t, 0.5 * g * g]
        return [t ** 3 / 6.0, 2.0 / 3.0 - g * g * (1.0 - 0.5 * g), 2.0 / 3.0 - t * t * (1.0 - 0.5 * t), g ** 3 / 6.0]

    def _nodes(self, r0):
        """(node weight, linear index, basis weight) terms of the lines r0 .. r0 + chunk."""
        s, w, n = self.s[r0:r0 + self.chunk], self.w[r0:r0 + self.chunk], self.n
        W = 0.5 * (n + 1)
        ts, lo, hi = [], None, None
        for e in range(3):
            kn = torch.arange(self.dims[e] + n + 1, device="cuda", dtype=torch.float64) - W
            d = kn[None, :] - s[:, e:e + 1]
            # a line that does not move along the axis meets no plane: all of them lie far behind or ahead
            t = torch.where(w[:, e:e + 1] == 0.0, torch.where(d < 0.0, -1.0e9, 1.0e9), d / w[:, e:e + 1])
            ends = torch.stack([t[:, 0], t[:, -1]])
            a, b = ends.min(dim=0).values, ends.max(dim=0).values
            lo, hi = (a, b) if lo is None else (torch.maximum(lo, a), torch.minimum(hi, b))
            ts.append(t)
        hi = torch.maximum(lo, hi)
        t = torch.cat(ts, dim=1)
        t = torch.minimum(torch.maximum(t, lo[:, None]), hi[:, None]).sort(dim=1).values
        h, m = 0.5 * (t[:, 1:] - t[:, :-1]), 0.5 * (t[:, 1:] + t[:, :-1])
        nx, ny, nz = self.dims
        for xq, wq in zip(self.x, self.wt):
            tq = m + xq * h
            cells, wts = [], []
            for e in range(3):
                v = s[:, e:e + 1] + tq * w[:, e:e + 1] + W
                c = v.floor()
                wts.append(self._weights(n, v - c))
                cells.append(c.long() - n)
            for k in range(n + 1):
                z = cells[2] + k
                for j in range(n + 1):
                    y = cells[1] + j
                    wy = wts[2][k] * wts[1][j] * (h * wq)
                    yz = (z >= 0) & (z < nz) & (y >= 0) & (y < ny)
                    base = (z * ny + y) * nx
                    for i in range(n + 1):
                        x = cells[0] + i
                        ok = yz & (x >= 0) & (x < nx)
                        yield torch.where(ok, base + x, 0), torch.where(ok, wy * wts[0][i], 0.0)

    def forward(self, c):
        flat = c.double().reshape(-1)
        out = torch.zeros(self.s.shape[0], dtype=torch.float64, device="cuda")
        for r0 in range(0, self.s.shape[0], self.chunk):
            for idx, wt in self._nodes(r0):
                out[r0:r0 + self.chunk] += (flat[idx] * wt).sum(dim=1)
        return out.reshape(self.shape)

    def adjoint(self, y):
        flat = y.double().reshape(-1)
        out = torch.zeros(self.dims[0] * self.dims[1] * self.dims[2], dtype=torch.float64, device="cuda")
        for r0 in range(0, self.s.shape[0], self.chunk):
            yr = flat[r0:r0 + self.chunk, None]
            for idx, wt in self._nodes(r0):
                out.index_add_(0, idx.reshape(-1), (wt * yr).reshape(-1))
        return out.reshape(self.dims[2], self.dims[1], self.dims[0])


def _exact_network(case, seed):
    p = torch.tensor(_network(seed), device="cuda", dtype=torch.float64).requires_grad_()
    feat, label = _batch(case, seed)
    h, o = feat.double(), 0
    for fan_in, fan_out in ((5, 64), (64, 64), (64, 64), (64, 1)):
        wt = p[o:o + fan_in * fan_out].reshape(fan_out, fan_in)
        o += fan_in * fan_out
        h = h @ wt.T + p[o:o + fan_out]
        o += fan_out
        if fan_out > 1:
            h = torch.nn.functional.silu(h)
    loss = (h[:, 0] - label.double()).square().mean()
    (g,) = torch.autograd.grad(loss, p)
    return g, loss.detach().reshape(1)


def exact(case, seed):
    op = case["op"]
    if op == "learned-gradient":
        return _exact_network(case, seed)
    if op.startswith("learned"):
        return None
    rays = case["rays"] if case["kind"] == "rays" else (case["views"] + case.get("tilt", 0)) * case["nu"] * case["nv"]
    knots = sum(_dims(case)) + 3 * (case["degree"] + 1)
    calls = {"gradient": 3, "adjoint": 2, "cgls": 2 + 3 * case.get("iters", 0)}.get(op, 1)
    if float(rays) * knots * ((3 * case["degree"] + 2) // 2) * (case["degree"] + 1) ** 3 * calls > EXACT_LIMIT:
        return None
    A = _Exact(case, seed)
    if op == "forward":
        return A.forward(_coefficients(case, seed))
    y = _projection(A.shape, seed)
    if op == "adjoint":
        return A.adjoint(y)
    if op == "gradient":
        p = A.forward(_coefficients(case, seed))
        return p, A.adjoint(p - y.double())
    x, r = 0.0, y.double()
    s = A.adjoint(r)
    p, gamma = s, (s * s).sum()
    for _ in range(case["iters"]):
        q = A.forward(p)
        alpha = gamma / (q * q).sum()
        x, r = x + alpha * p, r - alpha * q
        s = A.adjoint(r)
        p, gamma = s + (s * s).sum() / gamma * p, (s * s).sum()
    return x
