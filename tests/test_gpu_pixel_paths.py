"""Degree 0 on the automatic path: strip or general kernels by the number of
lines and their spacing, the same in plans, one-shot calls and batches; both
give the same results.  (Forward projections are deterministic and the two
families round differently, so equal bits tell which one ran.)"""
import math

import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"
G = torch.Generator


def _beam(kind, n, views, bins, ddet):
    v = ((torch.arange(views, dtype=torch.float64) + 0.37) * (math.pi / views)).float().to(DEV)
    det0 = -0.5 * (bins - 1) * ddet
    if kind == "parallel":
        return sp.Lines.parallel(v, bins, det0, ddet)
    return sp.Lines.fan(2.0 * v, 2.0 * n, 1.0 * n, bins, det0, ddet)


def _list(m, n):
    g = G(DEV).manual_seed(m)
    u = torch.rand((2, m), device=DEV, generator=g)
    return sp.Lines.theta_y(u[0] * 6.0 - 3.0, (u[1] - 0.5) * 1.3 * n)


CASES = [   # grid, lines, forward and adjoint on the strip kernels
    ((64, 64), lambda: _beam("parallel", 64, 30, 96, 1.0), False, False),
    ((64, 64), lambda: _beam("parallel", 64, 180, 96, 1.0), False, True),
    ((300, 512), lambda: _beam("parallel", 512, 30, 768, 1.0), True, True),
    ((512, 512), lambda: _beam("fan", 512, 60, 512, 2.9), True, True),
    ((512, 512), lambda: _beam("fan", 512, 60, 512, 4.4), True, False),
    ((512, 512), lambda: _beam("fan", 512, 60, 512, 4.6), False, False),
    ((512, 512), lambda: _beam("parallel", 512, 300, 96, 4.0), False, False),
    ((512, 512), lambda: _beam("parallel", 512, 700, 33, 1.0), False, False),
    ((200, 256), lambda: _list(1000, 256), False, False),
    ((200, 256), lambda: _list(40000, 256), True, False),
]


@pytest.mark.parametrize("size,make,fwd,adj", CASES)
def test_which_kernels_run(size, make, fwd, adj):
    nx, ny = size
    grid, lines = sp.Grid(nx, ny, 0), make()
    gen = G(DEV).manual_seed(5)
    coef = torch.rand((ny, nx), device=DEV, generator=gen) - 0.3
    p = torch.rand(lines.m, device=DEV, generator=gen) - 0.3
    plan = sp.Plan(grid, lines)
    auto, back = plan.fwd(coef), plan.adj(p)
    plan.set_paths(1, 1)
    strip, sback = plan.fwd(coef), plan.adj(p)
    plan.set_paths(2, 2)
    general, gback = plan.fwd(coef), plan.adj(p)
    assert torch.equal(auto, strip if fwd else general) and not torch.equal(strip, general)
    # sums of at most 2048 rounded terms: 1e-6 of the norm
    assert float((strip - general).norm() / general.norm()) < 1e-6
    assert float((sback - gback).norm() / gback.norm()) < 1e-6
    closer = (back - sback).norm() < (back - gback).norm()
    assert bool(closer) == adj
    assert torch.equal(sp.spline_project_fwd(grid, coef, lines), auto)
    once = sp.spline_project_adj(grid, p, lines)
    assert float((once - back).norm() / back.norm()) < 1e-6
    batch = sp.Batch([grid, grid], [lines, lines])
    for a in batch.fwd([coef, coef]):
        assert torch.equal(a, auto)
    for a in batch.adj([p, p]):
        assert float((a - back).norm() / back.norm()) < 1e-6
    plan.close()
    batch.close()
