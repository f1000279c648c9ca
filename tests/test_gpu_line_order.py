"""The chunk order of free line lists (order.cu) around the sizes of its blocks
(2048 lines per block and pass, 256 per scan step): every line projected once
whatever its place in the list, lines that miss the grid included.  A line's
value does not depend on the lines it shares a chunk with, so a permuted list
must give the permuted projection bit for bit; against the general path at the
parity bar (relative L2 1e-5)."""
import numpy as np
import pytest

from _geom import rel_l2

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"
TOL = 1e-5


def _project(grid, th, yy, coef, paths):
    plan = sp.Plan(grid, sp.Lines.theta_y(torch.from_numpy(th).to(DEV), torch.from_numpy(yy).to(DEV)), prepare=True)
    plan.set_paths(*paths)
    out = torch.full((len(th),), float("nan"), device=DEV)
    plan.fwd(coef, out)
    p = torch.cos(3.0 * torch.from_numpy(th).to(DEV)) + torch.from_numpy(yy).to(DEV) / 64.0
    back = plan.adj(p)
    plan.close()
    return out.cpu().numpy(), back.cpu().numpy()


@pytest.mark.parametrize("m", [1, 33, 2047, 2048, 2049, 4097, 600_011])
def test_permuted_lists(m):
    rng = np.random.default_rng(m)
    th = rng.uniform(-7.0, 7.0, m).astype(np.float32)
    yy = rng.uniform(-45.0, 45.0, m).astype(np.float32)     # a grid of 48 x 40: some lines miss it
    coef = torch.from_numpy(rng.standard_normal((40, 48)).astype(np.float32)).to(DEV)
    grid = sp.Grid(48, 40, 2)
    fwd, adj = _project(grid, th, yy, coef, (1, 1))
    assert np.isfinite(fwd).all()
    assert m == 1 or (fwd[np.abs(yy) > 36.0] == 0.0).all()  # beyond the grid's corners and the support
    perm = rng.permutation(m)
    fwd2, adj2 = _project(grid, th[perm], yy[perm], coef, (1, 1))
    assert np.array_equal(fwd2, fwd[perm])
    assert rel_l2(adj2, adj) < TOL
    ref_f, ref_a = _project(grid, th, yy, coef, (2, 2))
    if np.abs(ref_f).max() > 0:
        assert rel_l2(fwd, ref_f) < TOL and rel_l2(adj, ref_a) < TOL
