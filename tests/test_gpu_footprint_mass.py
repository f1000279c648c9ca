"""Errors of the strip kernels' footprints that are alike for all lines: each
line of an image of ones is off by FP32 rounding, 3e-8 to 6e-8, but the mean over
many directions is not, since backprojections of small residuals add it up.
Bound: 6000 independent lines leave 6e-8 / sqrt(6000) = 8e-10 of it; 5e-9 allows
that six times."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_the_mean_error_over_directions(degree):
    n, m = 64, 6000
    rng = np.random.default_rng(degree)
    th = rng.uniform(-3.1, 3.1, m).astype(np.float32)
    yy = rng.uniform(-24.0, 24.0, m).astype(np.float32)
    lines = sp.Lines.theta_y(torch.from_numpy(th).to(DEV), torch.from_numpy(yy).to(DEV))
    plan = sp.Plan(sp.Grid(n, n, degree, 1.0), lines)
    plan.set_paths(1, 1)
    got = plan.fwd(torch.ones((n, n), device=DEV)).double().cpu().numpy()
    plan.close()
    ref = oracle.forward(oracle.Grid(n, n, degree, 1.0), np.ones((n, n)), th.astype(np.float64), yy.astype(np.float64))
    assert abs((got - ref).mean()) < 5e-9 * ref.mean()
