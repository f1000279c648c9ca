"""Strip kernels where their cases meet: directions at and beside the slopes
b/a at which a breakpoint of the footprint passes a grid column (the base
interval and the number of knot groups change there), strips cut into several
slabs, groups of lines too wide for one strip row, rows and columns that are
not multiples of the row block or of 16 bytes.  Against the FP64 oracle at the
parity bar of the projector (relative L2 1e-5)."""
import math

import numpy as np
import pytest

import oracle
import workloads
from _geom import rel_l2

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"
TOL = 1e-5


def _check(grid, og, lines, th, yy, coef, seed):
    plan = sp.Plan(grid, lines, prepare=True)
    plan.set_paths(1, 1)
    got = plan.fwd(torch.from_numpy(coef).to(DEV)).cpu().numpy()
    assert rel_l2(got, oracle.forward(og, coef.astype(np.float64), th, yy)) < TOL
    p = np.random.default_rng(seed).uniform(-1.0, 1.0, lines.m).astype(np.float32)
    back = plan.adj(torch.from_numpy(p).to(DEV)).cpu().numpy()
    assert rel_l2(back, oracle.adjoint(og, p.astype(np.float64), th, yy)) < TOL
    plan.close()


SLOPES = [0.0, 1e-8, 1e-6, 1e-4, 0.01, 0.2, 0.25, 1 / 3, 0.4, 0.5, 2 / 3, 0.75, 0.9, 1.0]


@pytest.mark.parametrize("degree,basis", [(0, 0), (1, 0), (2, 0), (3, 0), (1, 1)])
def test_slopes_where_the_knots_change_columns(degree, basis):
    nx, ny = 38, 45
    th, yy = [], []
    for k, s in enumerate(SLOPES):
        for eps in (0.0, 3e-6, -3e-6, 0.02):
            base = math.atan(s) + eps
            t = [base, math.pi / 2 - base, math.pi / 2 + base, math.pi - base][k % 4]
            if degree == 0 and abs(math.sin(2 * t)) < 1e-5:
                t += 1e-3           # lines along pixel edges have no single value
            th += [t] * 41
            yy += list(np.linspace(-24.0, 24.0, 41) + 0.013 * k)
    th, yy = np.array(th, dtype=np.float32), np.array(yy, dtype=np.float32)
    lines = sp.Lines.theta_y(torch.from_numpy(th).to(DEV), torch.from_numpy(yy).to(DEV))
    coef = np.ascontiguousarray(workloads.ellipse_phantom(45, 8, 3, radius=15.0, axes=(2.0, 10.0))[:ny, :nx])
    _check(sp.Grid(nx, ny, degree, 1.0, basis=basis), oracle.Grid(nx, ny, degree, 1.0, basis=basis), lines,
           th.astype(np.float64), yy.astype(np.float64), coef, degree)


@pytest.mark.parametrize("nx,ny,degree,n_det,ddet", [
    (24, 1503, 3, 40, 0.7),       # several slabs, rows not in whole blocks
    (1502, 24, 2, 33, 0.9),       # the same on the transposed image, ragged chunk
    (260, 64, 3, 70, 4.5),        # 32 neighbouring lines wider than a strip row
    (64, 61, 1, 5, 11.0),         # few lines, far apart
])
def test_slabs_and_wide_groups(nx, ny, degree, n_det, ddet):
    view = (np.array([0.02, 0.4, 1.1, math.pi / 2 - 0.01, 2.0, 2.9])).astype(np.float32)
    det0 = float(np.float32(-0.5 * (n_det - 1) * ddet))
    ddet = float(np.float32(ddet))
    lines = sp.Lines.parallel(torch.from_numpy(view).to(DEV), n_det, det0, ddet)
    th, yy = oracle.lines_parallel(view.astype(np.float64), n_det, det0, ddet)
    rng = np.random.default_rng(nx)
    coef = rng.uniform(0.0, 1.0, (ny, nx)).astype(np.float32)
    _check(sp.Grid(nx, ny, degree, 1.0), oracle.Grid(nx, ny, degree, 1.0), lines, th, yy, coef, 5)


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_a_line_does_not_depend_on_its_chunk(degree):
    # one fan view whole, and its bins as lists of other lengths and mates
    n, n_det = 72, 100
    view = torch.tensor([0.71], device=DEV)
    grid = sp.Grid(n, n, degree, 1.0)
    coef = torch.from_numpy(workloads.ellipse_phantom(n, 8, 4, radius=24.0, axes=(2.0, 14.0))).to(DEV)
    whole = sp.spline_project_fwd(grid, coef, sp.Lines.parallel(view, n_det, -49.5, 1.0))
    for first, count in ((0, 1), (7, 33), (40, 60), (64, 3)):
        part = sp.spline_project_fwd(grid, coef, sp.Lines.parallel(view, count, -49.5 + first, 1.0))
        assert torch.equal(part, whole[first:first + count])


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_a_nonfinite_coefficient_reaches_its_lines_only(degree):
    # the kernels may multiply nodes just beyond a row's support by 0: lines
    # whose sum is not finite are taken again over their support alone
    n = 40
    view = np.array([0.0, 0.3, math.pi / 4, 1.2, 2.2], dtype=np.float32)
    lines = sp.Lines.parallel(torch.from_numpy(view).to(DEV), 64, -31.7, 1.0)
    th, yy = oracle.lines_parallel(view.astype(np.float64), 64, float(np.float32(-31.7)), 1.0)
    og = oracle.Grid(n, n, degree, 1.0)
    mask = np.zeros((n, n))
    mask[21, 17] = 1.0
    touched = oracle.forward(og, mask, th, yy)
    coef = workloads.ellipse_phantom(n, 8, 4, radius=14.0, axes=(2.0, 8.0))
    ref = oracle.forward(og, coef.astype(np.float64), th, yy)
    for bad in (np.nan, np.inf):
        c = coef.copy()
        c[21, 17] = bad
        got = sp.spline_project_fwd(sp.Grid(n, n, degree, 1.0), torch.from_numpy(c).to(DEV), lines).cpu().numpy()
        assert not np.any(np.isfinite(got[touched > 1e-5]))     # (the footprint vanishes smoothly at its ends)
        clear = touched == 0.0
        assert clear.any() and np.all(np.isfinite(got[clear]))
        assert rel_l2(got[clear], ref[clear]) < TOL


def test_plan_builds_footprint_tables_for_the_paths_that_read_them():
    # the strip kernels read none; a plan that switches to the other kernels
    # after prepare, prepares again with new angles, or captures a projection,
    # gets the tables of its lines
    n = 48
    view = torch.linspace(0.0, 3.0, 31, device=DEV)
    grid, lines = sp.Grid(n, n, 3, 1.0), sp.Lines.parallel(view, 70, -34.5, 1.0)
    coef = torch.from_numpy(workloads.ellipse_phantom(n, 8, 4, radius=16.0, axes=(2.0, 9.0))).to(DEV)
    p = torch.rand(lines.m, device=DEV, generator=torch.Generator(DEV).manual_seed(1))

    def close(a, b):
        return float((a - b).norm() / b.norm()) < 2e-6

    plan = sp.Plan(grid, lines)
    f, b = plan.fwd(coef), plan.adj(p)
    for adj_path in (2, 3):
        plan.set_paths(2, adj_path)
        assert close(plan.fwd(coef), f) and close(plan.adj(p), b)
    view.add_(0.21)
    plan.prepare()
    g = sp.spline_project_fwd(grid, coef, lines)
    assert close(plan.fwd(coef), g) and not close(g, f)
    fresh = sp.Plan(grid, lines)
    fresh.set_paths(2, 2)
    out = torch.empty(lines.m, device=DEV)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        fresh.fwd(coef, out)
    direct = fresh.fwd(coef).clone()      # before the graph has run
    graph.replay()
    torch.cuda.synchronize()
    assert close(direct, g) and torch.equal(direct, out)
    plan.close()
    fresh.close()
