"""Degree-0 adjoint of a sinogram with one line far above the others: pixels that
the strong line does not meet keep FP32 accuracy, on every kernel path and in
a batch.  Bound: sums of at most 80 terms and footprints good to 2e-7 stay
within 80 2^-24 + 2e-7 = 5e-6 of the largest such pixel."""
import math

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _lines(kind, n, bins):
    view = ((np.arange(40) + 0.4) * (math.pi / 40)).astype(np.float32)
    det0 = float(np.float32(-0.5 * (bins - 1)))
    th, yy = oracle.lines_parallel(view.astype(np.float64), bins, det0, 1.0)
    if kind == "parallel":
        return sp.Lines.parallel(torch.from_numpy(view).to(DEV), bins, det0, 1.0), th, yy
    th, yy = th.astype(np.float32), yy.astype(np.float32)
    return (sp.Lines.theta_y(torch.from_numpy(th).to(DEV), torch.from_numpy(yy).to(DEV)),
            th.astype(np.float64), yy.astype(np.float64))


@pytest.mark.parametrize("kind", ["parallel", "list"])
@pytest.mark.parametrize("run", [0, 1, 2, "batch"])
def test_pixels_beside_a_strong_line(run, kind):
    n, bins, strong = 61, 90, 17 * 90 + 44
    lines, th, yy = _lines(kind, n, bins)
    og, grid = oracle.Grid(n, n, 0, 1.0), sp.Grid(n, n, 0, 1.0)
    p = np.random.default_rng(3).uniform(0.5, 1.5, lines.m).astype(np.float32)
    p[strong] = 1e7
    only = np.zeros(lines.m)
    only[strong] = 1.0
    weak = oracle.adjoint(og, only, th, yy) == 0.0
    ref = oracle.adjoint(og, p.astype(np.float64), th, yy)
    pt = torch.from_numpy(p).to(DEV)
    if run == "batch":
        batch = sp.Batch([grid], [lines])
        got = batch.adj([pt])[0].cpu().numpy()
    else:
        plan = sp.Plan(grid, lines)
        plan.set_paths(0, run)
        got = plan.adj(pt).cpu().numpy()
    assert weak.sum() > 0.9 * n * n
    assert np.abs(got - ref)[weak].max() < 5e-6 * ref[weak].max()
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
