"""Degree-0 lines within a float's step of an axis that run along pixel edges:
their share of the two columns changes over ramps far narrower than an ulp of the
offset, on every kernel path the definition's."""
import math

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("path", [0, 1, 2])
@pytest.mark.parametrize("nx,ny,h", [(33, 40, 1.0), (90, 33, 0.5), (300, 16, 1.0)])
def test_views_beside_the_axes(nx, ny, h, path):
    # (the angles are those of float32: sin(fl(pi)) = -8.7e-8 and so on)
    view = np.array([math.pi, math.pi / 2, -math.pi / 2, 1e-7, 1.1e-6, 1e-5, 3e-4, math.pi / 2 + 1e-6], dtype=np.float32)
    bins = 2 * max(nx, ny) + 3
    det0, ddet = -0.25 * h * (bins - 1), 0.5 * h           # every pixel centre and edge
    lines = sp.Lines.parallel(torch.from_numpy(view).to(DEV), bins, det0, ddet)
    th, yy = oracle.lines_parallel(view.astype(np.float64), bins, det0, ddet)
    og = oracle.Grid(nx, ny, 0, h)
    rng = np.random.default_rng(nx)
    coef, p = rng.uniform(-1.0, 1.0, (ny, nx)).astype(np.float32), rng.uniform(-1.0, 1.0, lines.m).astype(np.float32)
    plan = sp.Plan(sp.Grid(nx, ny, 0, h), lines)
    plan.set_paths(path, path)
    sino = plan.fwd(torch.from_numpy(coef).to(DEV)).cpu().numpy()
    back = plan.adj(torch.from_numpy(p).to(DEV)).cpu().numpy()
    plan.close()
    # the projector's bar, for every line and pixel (a row of a line whose ramp is
    # narrower than the FP64 definition resolves can differ: b above 4e-8 is not)
    ref = oracle.forward(og, coef.astype(np.float64), th, yy)
    assert np.abs(sino - ref).max() < 1e-5 * np.abs(ref).max()
    ref = oracle.adjoint(og, p.astype(np.float64), th, yy)
    assert np.abs(back - ref).max() < 1e-5 * np.abs(ref).max()
