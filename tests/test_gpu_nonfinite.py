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
        if path != 2 or degree == 0:   # (the other general kernels multiply candidates beyond the support by 0)
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


@pytest.mark.parametrize("path", [0, 1, 2])
@pytest.mark.parametrize("degree,basis", [(0, 0), (1, 0), (2, 0), (3, 0), (1, 1)])
def test_a_line_sees_only_the_nodes_it_meets(degree, basis, path):
    # a coefficient of any size leaves every line that does not meet it as it
    # is, bit for bit; a line that misses the support of every basis gives 0
    og, grid = oracle.Grid(N, N, degree, 1.0, basis=basis), sp.Grid(N, N, degree, 1.0, basis=basis)
    for kind in ("parallel", "list"):
        lines, th, yy = _scan(kind)
        plan = sp.Plan(grid, lines)
        plan.set_paths(path, 0)
        coef = torch.rand((N, N), device=DEV, generator=torch.Generator(DEV).manual_seed(2)) + 0.5
        missed = oracle.forward(og, np.ones((N, N)), th, yy) == 0.0
        got = plan.fwd(coef).cpu().numpy()
        assert missed.sum() > 20 and np.all(got[missed] == 0.0) and np.all(got[~missed] >= 0.0)
        for j, i in ((21, 17), (0, 0), (39, 20)):
            mask = np.zeros((N, N))
            mask[j, i] = 1.0
            clear = oracle.forward(og, mask, th, yy) == 0.0
            c = coef.clone()
            c[j, i] = 0.0
            without = plan.fwd(c).cpu().numpy()
            for big in (1e30, np.inf if path != 2 or degree == 0 else 1e38):
                c[j, i] = big
                assert np.array_equal(plan.fwd(c).cpu().numpy()[clear], without[clear])
        plan.close()
