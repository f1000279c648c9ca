"""Infinite coefficients and sums that overflow: the forward gives infinities of
the right sign where FP32 sums of positive terms do."""
import math

import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"
N = 40


def _scan(kind):
    view = np.array([0.01, 0.3, math.pi / 4 + 0.01, 1.2, 2.2], dtype=np.float32)
    th, yy = oracle.lines_parallel(view.astype(np.float64), 64, float(np.float32(-31.7)), 1.0)
    if kind == "parallel":
        return sp.Lines.parallel(torch.from_numpy(view).to(DEV), 64, -31.7, 1.0), th, yy
    return sp.Lines.theta_y(torch.from_numpy(th).float().to(DEV), torch.from_numpy(yy).float().to(DEV)), th, yy


@pytest.mark.parametrize("kind", ["parallel", "list"])
@pytest.mark.parametrize("path", [0, 1, 2])
@pytest.mark.parametrize("degree,basis", [(0, 0), (1, 1)])
def test_an_infinite_coefficient(degree, basis, path, kind):
    lines, th, yy = _scan(kind)
    mask = np.zeros((N, N))
    mask[21, 17] = 1.0
    touched = oracle.forward(oracle.Grid(N, N, degree, 1.0, basis=basis), mask, th, yy)
    plan = sp.Plan(sp.Grid(N, N, degree, 1.0, basis=basis), lines)
    plan.set_paths(path, 0)
    coef = workloads.ellipse_phantom(N, 8, 4, radius=14.0, axes=(2.0, 8.0)).copy()
    for bad in (np.inf, -np.inf, np.nan):
        coef[21, 17] = bad
        got = plan.fwd(torch.from_numpy(coef).to(DEV)).cpu().numpy()
        met = got[touched > 1e-3]       # (the footprint vanishes smoothly at its ends)
        assert met.size > 5 and (np.all(np.isnan(met)) if np.isnan(bad) else np.all(met == bad))
        if path != 2:   # (the general kernels multiply the candidates beyond the support by 0)
            assert np.all(np.isfinite(got[touched == 0.0]))
    plan.close()


@pytest.mark.parametrize("path", [0, 1, 2])
@pytest.mark.parametrize("degree,basis", [(0, 0), (1, 0), (2, 0), (3, 0), (1, 1)])
def test_sums_that_overflow(degree, basis, path):
    lines, th, yy = _scan("parallel")
    length = oracle.forward(oracle.Grid(N, N, degree, 1.0, basis=basis), np.ones((N, N)), th, yy)
    plan = sp.Plan(sp.Grid(N, N, degree, 1.0, basis=basis), lines)
    plan.set_paths(path, 0)
    for sign in (1.0, -1.0):
        got = plan.fwd(torch.full((N, N), sign * 3e38, device=DEV)).cpu().numpy()
        assert np.all(got[length > 1.5] == sign * np.inf)
    plan.close()
