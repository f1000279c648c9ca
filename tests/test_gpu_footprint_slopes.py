"""Footprint tables at and within a few float32 steps of the directions whose
breakpoints p a + q b coincide (b/a a ratio of small integers), against the
oracle.  Bound: a table holds polynomials of at most 8 FP32 coefficients, off by
up to 6e-7 together over all directions; 2e-6 allows that three times."""
import math

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _directions(steps=6):
    out = []
    for r in (1 / 5, 1 / 4, 1 / 3, 2 / 5, 1 / 2, 3 / 5, 2 / 3, 3 / 4, 4 / 5, 1.0):
        t = math.atan(r)
        for base in (t, math.pi / 2 - t, math.pi / 2 + t, math.pi - t, -t):
            v = np.float32(base)
            for _ in range(steps):
                v = np.nextafter(v, np.float32(-10))
            for _ in range(2 * steps + 1):
                out.append(v)
                v = np.nextafter(v, np.float32(10))
    return np.array(out, dtype=np.float32)


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_footprints_beside_coinciding_breakpoints(degree):
    th = np.repeat(_directions(), 40)
    w = 0.5 * (degree + 1) * (np.abs(np.cos(th.astype(np.float64))) + np.abs(np.sin(th.astype(np.float64))))
    y = (np.random.default_rng(degree).uniform(-1.0, 1.0, th.size) * w).astype(np.float32)
    got = sp.spline_footprint_eval(degree, torch.from_numpy(th).to(DEV), torch.from_numpy(y).to(DEV)).cpu().numpy()
    ref = np.array([oracle.footprint(degree, float(t), float(v)) for t, v in zip(th, y)])
    assert np.abs(got - ref).max() < 2e-6


@pytest.mark.parametrize("paths", [(1, 1), (2, 2), (2, 3)])
@pytest.mark.parametrize("degree", [1, 2, 3])
def test_views_beside_coinciding_breakpoints(degree, paths):
    n, bins = 30, 50
    view = _directions(1)
    grid, og = sp.Grid(n, n, degree, 1.0), oracle.Grid(n, n, degree, 1.0)
    lines = sp.Lines.parallel(torch.from_numpy(view).to(DEV), bins, -24.7, 1.0)
    th, yy = oracle.lines_parallel(view.astype(np.float64), bins, float(np.float32(-24.7)), 1.0)
    rng = np.random.default_rng(degree)
    coef, p = rng.uniform(0.0, 1.0, (n, n)).astype(np.float32), rng.uniform(0.0, 1.0, lines.m).astype(np.float32)
    plan = sp.Plan(grid, lines)
    plan.set_paths(*paths)
    sino = plan.fwd(torch.from_numpy(coef).to(DEV)).cpu().numpy()
    back = plan.adj(torch.from_numpy(p).to(DEV)).cpu().numpy()
    plan.close()
    ref = oracle.forward(og, coef.astype(np.float64), th, yy)
    # every line by itself, of about the size of the largest: the projector's bar
    assert np.abs(sino - ref).max() < 1e-5 * ref.max()
    ref = oracle.adjoint(og, p.astype(np.float64), th, yy)
    assert np.abs(back - ref).max() < 1e-5 * ref.max()
