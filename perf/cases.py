"""Workloads of the spline x-ray projector: what its users run, at the sizes
they run it.

A case is a dict of plain values.  Its "op" names the entry points one pass
goes through:

  oneshot   spline_project_fwd and spline_project_adj (no plan)
  step      a plan's prepare, fwd and adj (a new scan geometry every pass)
  fwd, adj  one direction of a prepared plan
  grad      autograd: a projection, a loss gradient and its backprojection
  cgls      Plan.cgls from zero, with the plan's row records kept
  batch     Batch.fwd and Batch.adj of uneven instances
  net       the warm-start network's forward on an image
  train     the network's forward and backward on a batch of images

and the rest its sizes: an nx x ny grid of spacing h and B-spline degree
`degree`, and the lines: "parallel" and "fan" beams of `views` x `bins`,
"chords" (point pairs on a circle) or "theta_y" lists of `bins` lines.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2503_20907_gb300 as sp
from paper_2503_20907_gb300 import warmstart

DEV = "cuda"


def _proj(name, op, kind, nx, ny, degree, views, bins, **more):
    c = {"name": name, "op": op, "kind": kind, "nx": nx, "ny": ny, "degree": degree, "views": views, "bins": bins,
         "h": 1.0, "ddet": 1.0}
    c.update(more)
    c["h"] = float(np.float32(c["h"]))      # as the library takes it
    return c


def listed():
    return [
        # the smallest call: 64 x 64 linear splines, 90 angles x 96 offsets,
        # one-shot entry points (quick looks, unit tests of a pipeline)
        _proj("oneshot_parallel64_linear", "oneshot", "parallel", 64, 64, 1, 90, 96),
        # the repository's benchmark step: a 512 x 512 cubic fan-beam scan
        _proj("step_fan512_cubic", "step", "fan", 512, 512, 3, 720, 768),
        # the warm start's geometry: sinograms of training phantoms
        _proj("fwd_parallel256_cubic", "fwd", "parallel", 256, 256, 3, 360, 384),
        # ragged sizes: rectangular grid with odd sides, odd bins, spacing
        # other than one
        _proj("adj_fan333x257_quadratic", "adj", "fan", 333, 257, 2, 501, 487, h=0.5, ddet=0.53),
        # learned reconstruction: gradient of a data term through the projector
        _proj("grad_fan256_linear", "grad", "fan", 256, 256, 1, 360, 384),
        # the largest scan of the uneven batch's ranges, projections of a
        # prepared plan's geometry
        _proj("step_parallel1024_quadratic", "step", "parallel", 1024, 1024, 2, 1440, 1536),
        # arbitrary line lists: a million random chords through a 512 x 512 grid
        _proj("step_chords512_cubic", "step", "chords", 512, 512, 3, 1, 1000000),
        # pixel basis (degree 0), odd sizes
        _proj("grad_parallel501_pixels", "grad", "parallel", 501, 501, 0, 367, 751),
        # iterative reconstruction: the first CGLS iterations at 256 x 256
        _proj("cgls_parallel256_cubic", "cgls", "parallel", 256, 256, 3, 360, 384, iters=4),
        # uneven instances projected together (sizes 128..1024, all degrees,
        # all kinds of lines)
        {"name": "batch8_uneven", "op": "batch", "first": 0, "count": 8, "scale": 0.7},
        # warm start at test time: one 256 x 256 image
        {"name": "net_1x256", "op": "net", "images": 1, "nx": 256, "ny": 256},
        # training step of the warm start: a batch of eight
        {"name": "train_8x256", "op": "train", "images": 8, "nx": 256, "ny": 256},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_lines(rng, n):
    """Kind, views and bins of a scan of an image about n nodes wide."""
    kind = rng.choice(["parallel", "parallel", "fan", "fan", "fan", "chords", "theta_y"])
    if kind in ("chords", "theta_y"):
        return kind, 1, _logint(rng, 10 * n, 2000 * n)
    return kind, _logint(rng, 0.35 * n + 20, 1.4 * n + 20), int(n * rng.uniform(1.3, 1.6))


def draw(rng):
    op = rng.choice(["oneshot", "step", "step", "fwd", "fwd", "adj", "adj", "grad", "cgls", "batch", "net", "train"])
    if op == "net":
        return {"op": op, "images": 1, "nx": _logint(rng, 96, 512), "ny": _logint(rng, 96, 512)}
    if op == "train":
        return {"op": op, "images": rng.randint(2, 12), "nx": rng.randint(96, 300), "ny": rng.randint(96, 300)}
    if op == "batch":
        return {"op": op, "first": rng.randrange(8, 100000), "count": rng.randint(4, 10), "scale": rng.uniform(0.3, 0.6)}
    n = _logint(rng, 64, 384 if op == "cgls" else 1000)
    ny = n if rng.random() < 0.5 else max(33, int(n * rng.uniform(0.6, 1.0)))
    kind, views, bins = _draw_lines(rng, n)
    if op == "cgls":
        kind, views, bins = rng.choice(["parallel", "fan"]), int(1.4 * n), int(1.5 * n)
    h = rng.choice([1.0, 1.0, 0.5, 0.8])
    c = _proj(None, op, kind, n, ny, rng.choice([0, 1, 2, 3, 3]), views, bins, h=h, ddet=h * rng.uniform(0.85, 1.2))
    del c["name"]
    if op == "cgls":
        c["degree"] = rng.choice([1, 2, 3])
        c["iters"] = rng.randint(2, 4)
    return c


# ------------------------------------------------------------------ geometry
def _instances(case):
    """The scans of a batch: sizes log-uniform over 128..1024 times the scale,
    every eighth a list of chords."""
    out = []
    for i in range(case["first"], case["first"] + case["count"]):
        rng = random.Random(7919 * i + 13)
        n = max(32, int(round(math.exp(rng.uniform(math.log(128), math.log(1024))) * case["scale"])))
        degree = i % 4
        if i % 8 == 7:
            kind, views, bins = "chords", 1, int(rng.uniform(1e5, 1e6) * case["scale"] ** 2)
        else:
            kind = rng.choice(["parallel", "fan"])
            views, bins = int(rng.randint(180, 1440) * case["scale"]), int(round(1.5 * n))
        out.append(_proj(f"i{i}", "batch", kind, n, n, degree, views, bins))
    return out


def _extent(c):
    return max(c["nx"], c["ny"]) * c["h"]


def _scan(c, seed, device):
    """Float32 line parameters of a scan (what the user's program holds)."""
    g = torch.Generator(device=device).manual_seed(seed * 1009 + 7)
    kind, m = c["kind"], c["bins"]
    if kind in ("parallel", "fan"):
        span = math.pi if kind == "parallel" else 2.0 * math.pi
        # scans start on the axis; those of the pixel basis beside it, where a
        # line along pixel edges has no single value
        jit = float(torch.rand(1, generator=g, device=device)) if c["degree"] == 0 else 0.0
        v = (torch.arange(c["views"], dtype=torch.float64, device=device) + jit) * (span / c["views"])
        return {"view": v.float()}
    u = torch.rand((2, m), generator=g, device=device, dtype=torch.float64)
    r = 0.75 * _extent(c)
    if kind == "chords":
        a0, a1 = 2.0 * math.pi * u[0], 2.0 * math.pi * u[1]
        return {"src": torch.stack([r * a0.cos(), r * a0.sin()], 1).float(),
                "dst": torch.stack([r * a1.cos(), r * a1.sin()], 1).float()}
    return {"theta": (2.0 * math.pi * u[0] - math.pi).float(), "y": ((2.0 * u[1] - 1.0) * 0.7 * _extent(c)).float()}


def _detector(c):
    """det0, ddet, dso, dod of a beam (bins centred on the axis)."""
    ddet = float(np.float32(c["ddet"]))
    det0 = float(np.float32(-0.5 * (c["bins"] - 1) * ddet))
    return det0, ddet, float(np.float32(1.953125 * _extent(c))), float(np.float32(0.9765625 * _extent(c)))


def _lines(c, s):
    det0, ddet, dso, dod = _detector(c)
    if c["kind"] == "parallel":
        return sp.Lines.parallel(s["view"], c["bins"], det0, ddet)
    if c["kind"] == "fan":
        return sp.Lines.fan(s["view"], dso, dod, c["bins"], det0, ddet)
    if c["kind"] == "chords":
        return sp.Lines.points(s["src"], s["dst"])
    return sp.Lines.theta_y(s["theta"], s["y"])


def _rays(c, s):
    """FP64 direction (dx, dy) and a point (px, py) of every line, flat."""
    d = {k: v.double() for k, v in s.items()}
    det0, ddet, dso, dod = _detector(c)
    if c["kind"] in ("parallel", "fan"):
        co, si = d["view"].cos()[:, None], d["view"].sin()[:, None]
        off = det0 + ddet * torch.arange(c["bins"], dtype=torch.float64, device=co.device)[None, :]
        if c["kind"] == "parallel":
            px, py = off * si, -off * co
            dx, dy = co.expand_as(px), si.expand_as(px)
        else:
            sx, sy = dso * co, dso * si
            vx, vy = -dod * co - off * si - sx, -dod * si + off * co - sy
            ln = (vx * vx + vy * vy).sqrt()
            dx, dy, px, py = vx / ln, vy / ln, sx.expand_as(vx), sy.expand_as(vx)
        return [t.reshape(-1) for t in (dx, dy, px, py)]
    if c["kind"] == "chords":
        v = d["dst"] - d["src"]
        v = v / v.norm(dim=1, keepdim=True)
        return [v[:, 0], v[:, 1], d["src"][:, 0], d["src"][:, 1]]
    co, si = d["theta"].cos(), d["theta"].sin()
    return [co, si, d["y"] * si, -d["y"] * co]


# ------------------------------------------------------------------ inputs
def _ellipses(c, seed, device, count=20):
    g = torch.Generator().manual_seed(seed * 31 + 5)
    u = torch.rand((count, 6), generator=g, dtype=torch.float64)
    s = min(c["nx"], c["ny"]) * c["h"] / 64.0
    r, a = 24.0 * s * u[:, 0].sqrt(), 2.0 * math.pi * u[:, 1]
    e = torch.stack([r * a.cos(), r * a.sin(), (2.0 + 14.0 * u[:, 2]) * s, (2.0 + 14.0 * u[:, 3]) * s,
                     math.pi * u[:, 4], -0.5 + 1.5 * u[:, 5]], 1)
    return e.to(device)


def _phantom(c, seed, device=DEV):
    """Coefficients: a random-ellipse phantom sampled at the nodes."""
    X = (torch.arange(c["nx"], dtype=torch.float64, device=device) - 0.5 * (c["nx"] - 1)) * c["h"]
    Y = (torch.arange(c["ny"], dtype=torch.float64, device=device) - 0.5 * (c["ny"] - 1)) * c["h"]
    out = torch.zeros((c["ny"], c["nx"]), dtype=torch.float64, device=device)
    for x0, y0, A, B, rot, w in _ellipses(c, seed, device).tolist():
        dx, dy = X[None, :] - x0, Y[:, None] - y0
        p = (dx * math.cos(rot) + dy * math.sin(rot)) / A
        q = (-dx * math.sin(rot) + dy * math.cos(rot)) / B
        out += w * (p * p + q * q <= 1.0)
    return out.float()


def _sinogram(c, s, seed, noise=0.01):
    """Measured data of the ellipse phantom: its chord lengths, and noise."""
    dx, dy, px, py = _rays(c, s)
    out = torch.zeros_like(dx)
    for x0, y0, A, B, rot, w in _ellipses(c, seed, dx.device).tolist():
        c1, s1 = math.cos(rot), math.sin(rot)
        n1, n2 = dy * c1 - dx * s1, -dy * s1 - dx * c1              # theta^perp in the ellipse's axes
        r2 = (A * n1) ** 2 + (B * n2) ** 2
        off = (px - x0) * dy - (py - y0) * dx
        out += w * 2.0 * A * B * (r2 - off * off).clamp_min(0.0).sqrt() / r2
    g = torch.Generator(device=out.device).manual_seed(seed * 17 + 3)
    sc = noise * float(out.abs().max().clamp_min(1e-6))
    return (out + sc * torch.randn(out.shape, generator=g, device=out.device, dtype=torch.float64)).float()


def _images(case, seed):
    """Scaled backprojections: blurred noisy phantoms [B][ny][nx], and targets."""
    c = {"nx": case["nx"], "ny": case["ny"], "h": 1.0}
    t = torch.stack([_phantom(c, seed * 64 + k) for k in range(case["images"])])
    z = torch.nn.functional.avg_pool2d(t[:, None].double(), 9, 1, 4)[:, 0]
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    return (z + 0.02 * torch.randn(z.shape, generator=g, device=DEV, dtype=torch.float64)).float(), t


def _grid(c):
    return sp.Grid(c["nx"], c["ny"], c["degree"], c["h"])


def prepare(case, seed):
    op = case["op"]
    if op in ("net", "train"):
        net, _ = warmstart.load_net(warmstart.DEFAULT_WEIGHTS, DEV)
        z, target = _images(case, seed)
        return {"case": case, "net": net, "z": z, "target": target}
    if op == "batch":
        inst = _instances(case)
        scans = [_scan(c, seed + k, DEV) for k, c in enumerate(inst)]
        batch = sp.Batch([_grid(c) for c in inst], [_lines(c, s) for c, s in zip(inst, scans)])
        coefs = [_phantom(c, seed + k) for k, c in enumerate(inst)]
        sinos = [_sinogram(c, s, seed + k) for k, (c, s) in enumerate(zip(inst, scans))]
        return {"case": case, "batch": batch, "coefs": coefs, "sinos": sinos,
                "sino_out": [torch.empty_like(p) for p in sinos], "coef_out": [torch.empty_like(x) for x in coefs]}
    s = _scan(case, seed, DEV)
    st = {"case": case, "grid": _grid(case), "lines": _lines(case, s), "coef": _phantom(case, seed),
          "sino": _sinogram(case, s, seed)}
    if op != "oneshot":
        st["plan"] = sp.Plan(st["grid"], st["lines"], records=(op == "cgls"))
    return st


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "oneshot":
        return [sp.spline_project_fwd(state["grid"], state["coef"], state["lines"]),
                sp.spline_project_adj(state["grid"], state["sino"], state["lines"])]
    if op == "step":
        state["plan"].prepare()
        return [state["plan"].fwd(state["coef"]), state["plan"].adj(state["sino"])]
    if op == "fwd":
        return state["plan"].fwd(state["coef"])
    if op == "adj":
        return state["plan"].adj(state["sino"])
    if op == "grad":
        x = state["coef"].detach().requires_grad_(True)
        p = sp.project(x, state["plan"])
        r = p - state["sino"]
        (0.5 * (r * r).sum()).backward()
        return [p.detach(), x.grad]
    if op == "cgls":
        # as a solve of a known number of iterations runs it
        return state["plan"].cgls(state["sino"], case["iters"], history=False)[0]
    if op == "batch":
        return [state["batch"].fwd(state["coefs"], state["sino_out"]),
                state["batch"].adj(state["sinos"], state["coef_out"])]
    net = state["net"]
    if op == "net":
        with torch.no_grad():
            return net(state["z"])
    for p in net.parameters():
        p.grad = None
    x0 = net(state["z"])
    loss = ((x0 - state["target"]) ** 2).mean()
    loss.backward()
    return [x0.detach(), loss.detach()] + [p.grad for p in net.parameters()]


# ------------------------------------------------------------------ work
def _pairs(c):
    """Nonzero (line, node) pairs of one projection: a line of length l in the
    grid meets about l (n+1) (|cos| + |sin|) / h nodes.  From a sample of the
    lines on the CPU."""
    sub = dict(c)
    if c["kind"] in ("parallel", "fan"):
        sub["views"] = min(c["views"], 64)
    else:
        sub["bins"] = min(c["bins"], 20000)
    dx, dy, px, py = (t.numpy() for t in _rays(sub, _scan(sub, 1, "cpu")))
    n = c["degree"] + 1
    t0, t1 = np.full(dx.shape, -1e30), np.full(dx.shape, 1e30)
    for d, p, size in ((dx, px, c["nx"]), (dy, py, c["ny"])):
        dd = np.where(np.abs(d) < 1e-12, 1e-12, d)
        a, b = (-0.5 * size * c["h"] - p) / dd, (0.5 * size * c["h"] - p) / dd
        t0, t1 = np.maximum(t0, np.minimum(a, b)), np.minimum(t1, np.maximum(a, b))
    per = np.maximum(t1 - t0, 0.0) * (np.abs(dx) + np.abs(dy)) * n / c["h"]
    return float(per.mean()) * c["views"] * c["bins"]


def _scan_bytes(c):
    per = {"parallel": 4 * c["views"], "fan": 4 * c["views"], "chords": 16 * c["bins"], "theta_y": 8 * c["bins"]}
    return per[c["kind"]]


def work(case):
    op = case["op"]
    if op in ("net", "train"):
        px = case["images"] * case["nx"] * case["ny"]
        per = 2 * 9 * sum(cin * cout for cin, cout, _, _ in warmstart.LAYERS)
        w = sum(9 * cin * cout + cout for cin, cout, _, _ in warmstart.LAYERS)
        if op == "net":
            return {"bytes": 8 * px + 4 * w, "flops": per * px}
        first = 2 * 9 * warmstart.LAYERS[0][0] * warmstart.LAYERS[0][1]   # no input gradient there
        return {"bytes": 12 * px + 8 * w, "flops": (3 * per - first) * px}
    if op == "batch":
        parts = [work(dict(c, op="fwd")) for c in _instances(case)] + [work(dict(c, op="adj")) for c in _instances(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    n, m = case["nx"] * case["ny"], case["views"] * case["bins"]
    flops = 2 * (2 * case["degree"] + 3) * _pairs(case)      # per direction: Horner, offset, accumulate
    if op in ("fwd", "adj"):
        return {"bytes": 4 * (n + m) + _scan_bytes(case), "flops": flops}
    if op == "cgls":
        k = case["iters"] + 1
        return {"bytes": 4 * (m + n) + _scan_bytes(case), "flops": 2 * k * flops}
    # both directions
    return {"bytes": 8 * (n + m) + _scan_bytes(case), "flops": 2 * flops}


# ------------------------------------------------------------------ exact
def _bspline(x, n):
    """Centred B-spline of degree n (unit knots)."""
    x = x.abs()
    if n == 0:
        return (x < 0.5).to(x.dtype)
    if n == 1:
        return (1.0 - x).clamp_min(0.0)
    if n == 2:
        return torch.where(x < 0.5, 0.75 - x * x, 0.5 * (1.5 - x).clamp_min(0.0) ** 2)
    return torch.where(x < 1.0, 2.0 / 3.0 - x * x + 0.5 * x ** 3, (2.0 - x).clamp_min(0.0) ** 3 / 6.0)


def _footprint(y, a, b, n):
    """phi(y) = int beta_a(y - b s) beta(s) ds for the line integral of the
    tensor B-spline across a line with |cos|, |sin| = a >= b: Gauss-Legendre on
    the pieces of the integrand between the knots of both factors."""
    m = n + 1
    x, w = np.polynomial.legendre.leggauss(m)
    out = torch.zeros_like(y)
    bs = b.clamp_min(1e-30)
    for k in range(m):
        lo = torch.full_like(y, -0.5 * m + k)
        # knots of the first factor are a (j - m/2) apart: at most one inside
        # the unit interval, since b <= a
        j = torch.floor((y - bs * lo) / a + 0.5 * m)
        cut = ((y - a * (j - 0.5 * m)) / bs).clamp(min=lo, max=lo + 1.0)
        for l0, l1 in ((lo, cut), (cut, lo + 1.0)):
            hw, mid = 0.5 * (l1 - l0), 0.5 * (l1 + l0)
            for xi, wi in zip(x.tolist(), w.tolist()):
                s = mid + xi * hw
                out += wi * hw * _bspline((y - b * s) / a, n) / a * _bspline(s, n)
    return out


def _pieces(a, b, n):
    """Per direction: sorted breakpoints [L][K+1] of phi in u = y + w and, for
    every piece, its polynomial in the local variable v in [-1, 1]
    [L][K][2n+2], interpolated at Chebyshev nodes."""
    m, nc = n + 1, 2 * n + 2
    p = torch.arange(m + 1, dtype=torch.float64, device=a.device)
    br = (p[None, :, None] * a[:, None, None] + p[None, None, :] * b[:, None, None]).reshape(len(a), -1)
    br = br.sort(dim=1).values
    lo, hi = br[:, :-1, None], br[:, 1:, None]
    v = torch.cos(math.pi * (2 * torch.arange(nc, dtype=torch.float64, device=a.device) + 1) / (2 * nc))
    y = 0.5 * (lo + hi) + 0.5 * (hi - lo) * v - 0.5 * br[:, -1:, None]
    f = _footprint(y, a[:, None, None], b[:, None, None], n)
    V = torch.linalg.inv(v[:, None] ** torch.arange(nc, dtype=torch.float64, device=a.device)[None, :])
    return br, f @ V.T


class _Exact:
    """The projector of a scan in FP64."""

    def __init__(self, c, seed):
        s = _scan(c, seed, DEV)
        self.c, self.n = c, c["degree"]
        self.dx, self.dy, self.px, self.py = _rays(c, s)
        self.lines = len(self.dx)
        self.per_view = c["bins"] if c["kind"] == "parallel" else 1

    def _blocks(self):
        """(lines, rows, flat node index, footprint, valid) over chunks of
        lines, mainly vertical and mainly horizontal ones apart."""
        c, n, h = self.c, self.n, self.c["h"]
        vert = self.dy.abs() >= self.dx.abs()
        K = 2 * n + 4
        for up in (True, False):
            idx = torch.nonzero(vert == up)[:, 0]
            nr, nq = (c["ny"], c["nx"]) if up else (c["nx"], c["ny"])
            step = max(1, int(1.2e7) // (nr * K))
            for i0 in range(0, len(idx), step):
                l = idx[i0:i0 + step]
                dx, dy, px, py = self.dx[l], self.dy[l], self.px[l] / h, self.py[l] / h
                a = torch.maximum(dx.abs(), dy.abs())
                b = torch.minimum(dx.abs(), dy.abs())
                tab = l // self.per_view
                ut, inv = torch.unique_consecutive(tab, return_inverse=True)
                first = torch.searchsorted(tab.contiguous(), ut.contiguous())
                br, poly = _pieces(a[first], b[first], n)
                br, pieces = br[inv], poly.shape[1]
                r = torch.arange(nr, dtype=torch.float64, device=l.device)
                rr = r - 0.5 * (nr - 1)
                # yt(row, col) = [(px - x) dy - (py - y) dx] / h = base + slope_r rr + kappa qq
                kap = -dy if up else dx
                base = px * dy - py * dx
                cross = (base[:, None] + (dx if up else -dy)[:, None] * rr[None, :]) / -kap[:, None]   # qq where yt = 0
                q0 = torch.floor(cross + 0.5 * (nq - 1)) - (K // 2 - 1)
                q = q0[:, :, None] + torch.arange(K, dtype=torch.float64, device=l.device)
                u = kap[:, None, None] * (q - 0.5 * (nq - 1) - cross[:, :, None]) + 0.5 * br[:, -1:, None]
                ok = (q >= 0) & (q <= nq - 1) & (u > 0) & (u < br[:, -1:, None])
                flat = u.reshape(len(l), -1)
                k = (torch.searchsorted(br.contiguous(), flat.contiguous(), right=True) - 1).clamp(0, pieces - 1)
                blo, bhi = br.gather(1, k), br.gather(1, k + 1)
                v = (2.0 * flat - blo - bhi) / (bhi - blo).clamp_min(1e-300)
                row = inv[:, None] * pieces + k
                pf = poly.reshape(-1, poly.shape[2])
                phi = pf[:, -1][row]
                for d in range(poly.shape[2] - 2, -1, -1):
                    phi = phi * v + pf[:, d][row]
                phi = torch.where(ok, phi.reshape(u.shape), torch.zeros((), dtype=torch.float64, device=l.device))
                qi = q.clamp(0, nq - 1).long()
                ri = r.long()[None, :, None]
                node = ri * nq + qi if up else qi * nr + ri
                yield l, node, phi

    def fwd(self, x):
        x = x.double().reshape(-1)
        out = torch.zeros(self.lines, dtype=torch.float64, device=x.device)
        for l, node, phi in self._blocks():
            out[l] = self.c["h"] * (x[node] * phi).sum(dim=(1, 2))
        return out

    def adj(self, p):
        p = p.double()
        out = torch.zeros(self.c["nx"] * self.c["ny"], dtype=torch.float64, device=p.device)
        for l, node, phi in self._blocks():
            out.index_add_(0, node.reshape(-1), (self.c["h"] * p[l][:, None, None] * phi).reshape(-1))
        return out.reshape(self.c["ny"], self.c["nx"])


def _exact_cost(c):
    return c["views"] * c["bins"] * max(c["nx"], c["ny"]) * (2 * c["degree"] + 4) * (2 * c["degree"] + 8)


_EXACT_MAX = 6.0e10   # about a dozen seconds of both directions


def _net64(net, z):
    """The network in FP64 with the BF16 weights it is defined with."""
    ws = [w.detach().to(torch.bfloat16).double().requires_grad_(True) for w in net.w]
    bs = [b.detach().double().requires_grad_(True) for b in net.b]
    x = z.double()[:, None]
    for w, b, (_, _, relu, dil) in zip(ws, bs, warmstart.LAYERS):
        x = torch.nn.functional.conv2d(x, w.permute(0, 3, 1, 2), b, padding=dil, dilation=dil)
        x = x.relu() if relu else x
    return z.double() + x[:, 0], ws, bs


def exact(case, seed):
    op = case["op"]
    if op in ("net", "train"):
        net, _ = warmstart.load_net(warmstart.DEFAULT_WEIGHTS, DEV)
        z, target = _images(case, seed)
        x0, ws, bs = _net64(net, z)
        if op == "net":
            return x0.detach()
        loss = ((x0 - target.double()) ** 2).mean()
        loss.backward()
        return [x0.detach(), loss.detach()] + [w.grad for w in ws] + [b.grad for b in bs]
    if op == "batch":
        inst = _instances(case)
        if sum(2 * _exact_cost(c) for c in inst) > 2 * _EXACT_MAX:
            return None
        E = [_Exact(c, seed + k) for k, c in enumerate(inst)]
        return [[e.fwd(_phantom(c, seed + k)) for k, (c, e) in enumerate(zip(inst, E))],
                [e.adj(_sinogram(c, _scan(c, seed + k, DEV), seed + k)) for k, (c, e) in enumerate(zip(inst, E))]]
    passes = {"fwd": 1, "adj": 1, "cgls": 2 * (case.get("iters", 0) + 1)}.get(op, 2)
    if passes * _exact_cost(case) > 2 * _EXACT_MAX:
        return None
    E = _Exact(case, seed)
    x, p = _phantom(case, seed), _sinogram(case, _scan(case, seed, DEV), seed)
    if op == "fwd":
        return E.fwd(x)
    if op == "adj":
        return E.adj(p)
    if op in ("oneshot", "step"):
        return [E.fwd(x), E.adj(p)]
    if op == "grad":
        q = E.fwd(x)
        return [q, E.adj(q - p.double())]
    # conjugate gradients on the normal equations from zero
    xk = torch.zeros((case["ny"], case["nx"]), dtype=torch.float64, device=DEV)
    r = p.double()
    s = E.adj(r)
    d, gam = s, (s * s).sum()
    for _ in range(case["iters"]):
        q = E.fwd(d)
        alpha = gam / (q * q).sum()
        xk, r = xk + alpha * d, r - alpha * q
        s = E.adj(r)
        new = (s * s).sum()
        d, gam = s + (new / gam) * d, new
    return xk
