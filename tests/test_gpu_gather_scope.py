"""Adjoint path 3 on geometries whose lines through a node are no neighbours in
their view: a fan with part of the grid beside or behind its source (lines go on
behind it), and bins that coincide."""
import math

import numpy as np
import pytest

import oracle
from _geom import rel_l2

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("dso,dod,cx,ddet", [(20.0, 30.0, 0.0, 1.0), (45.0, -12.0, 0.0, 0.7), (70.0, 20.0, 50.0, 1.1),
                                              (150.0, 60.0, 0.0, 0.0), (150.0, 60.0, 3.0, -0.9), (150.0, 60.0, 0.0, 0.9)])
def test_fans(degree, dso, dod, cx, ddet):
    nx, ny, bins = 60, 44, 75
    view = ((np.arange(17) + 0.3) * (2.0 * math.pi / 17)).astype(np.float32)
    dso, dod, ddet, det0 = (float(np.float32(v)) for v in (dso, dod, ddet, -0.5 * (bins - 1) * ddet + 0.2))
    lines = sp.Lines.fan(torch.from_numpy(view).to(DEV), dso, dod, bins, det0, ddet)
    th, yy = oracle.lines_fan(view.astype(np.float64), dso, dod, bins, det0, ddet)
    p = np.random.default_rng(degree).uniform(0.0, 1.0, lines.m).astype(np.float32)
    plan = sp.Plan(sp.Grid(nx, ny, degree, 1.0, cx, 0.0), lines)
    plan.set_paths(0, 3)
    got = plan.adj(torch.from_numpy(p).to(DEV)).cpu().numpy()
    plan.close()
    assert rel_l2(got, oracle.adjoint(oracle.Grid(nx, ny, degree, 1.0, cx, 0.0), p.astype(np.float64), th, yy)) < 1e-5


def test_parallel_bins_that_coincide():
    n, bins = 40, 50
    view = np.array([0.3, 1.2, 2.0], dtype=np.float32)
    lines = sp.Lines.parallel(torch.from_numpy(view).to(DEV), bins, 1.3, 0.0)
    th, yy = oracle.lines_parallel(view.astype(np.float64), bins, float(np.float32(1.3)), 0.0)
    p = np.random.default_rng(1).uniform(0.0, 1.0, lines.m).astype(np.float32)
    plan = sp.Plan(sp.Grid(n, n, 3), lines)
    plan.set_paths(0, 3)
    got = plan.adj(torch.from_numpy(p).to(DEV)).cpu().numpy()
    plan.close()
    assert rel_l2(got, oracle.adjoint(oracle.Grid(n, n, 3, 1.0), p.astype(np.float64), th, yy)) < 1e-5
