"""Degree-0 lines exactly along an axis: the column's or row's sum, on a pixel
edge half of each side's (half of one at the border), 0 beyond; the same among
lines that are not along an axis.  Integer pixels and values: exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _weights(offset, n):
    """Share of each of n pixels (centres -(n-1)/2 ...) in a line at this offset."""
    c = np.arange(n) - 0.5 * (n - 1)
    d = np.abs(c - offset)
    return np.where(d < 0.5, 1.0, np.where(d == 0.5, 0.5, 0.0))


@pytest.mark.parametrize("path", [0, 1, 2])
@pytest.mark.parametrize("nx,ny,h", [(40, 33, 1.0), (33, 70, 0.5), (64, 64, 1.0), (5, 515, 1.0)])
def test_axis_lines(nx, ny, h, path):
    rng = np.random.default_rng(nx + ny)
    coef = rng.integers(-8, 9, (ny, nx)).astype(np.float32)
    src, dst, W = [], [], []
    for k in range(2 * max(nx, ny) + 9):
        off = -0.25 * max(nx, ny) - 2.0 + 0.25 * k          # centres, edges and between, and misses
        for up in (1.0, -1.0):
            src.append((off, -1000.0 * up)), dst.append((off, 1000.0 * up))
            W.append(np.outer(np.ones(ny), _weights(off, nx)))
            src.append((-1000.0 * up, off)), dst.append((1000.0 * up, off))
            W.append(np.outer(_weights(off, ny), np.ones(nx)))
    W = np.array(W)
    order = rng.permutation(len(W))
    s, d = np.array(src)[order] * h, np.array(dst)[order] * h
    lines = sp.Lines.points(torch.from_numpy(s.astype(np.float32)).to(DEV), torch.from_numpy(d.astype(np.float32)).to(DEV))
    plan = sp.Plan(sp.Grid(nx, ny, 0, h), lines)
    plan.set_paths(path, path)
    got = plan.fwd(torch.from_numpy(coef).to(DEV)).cpu().numpy()
    assert np.array_equal(got, h * np.einsum("lji,ji->l", W[order], coef))
    p = rng.integers(-8, 9, len(W)).astype(np.float32)
    back = plan.adj(torch.from_numpy(p).to(DEV)).cpu().numpy()
    assert np.array_equal(back, h * np.einsum("lji,l->ji", W[order], p))
    plan.close()


@pytest.mark.parametrize("path", [0, 1, 2])
def test_axis_views_of_a_scan(path):
    # a parallel view at angle 0 (its lines run along x1) among others
    n, bins = 48, 101
    rng = np.random.default_rng(7)
    coef = rng.integers(-8, 9, (n, n)).astype(np.float32)
    view = torch.tensor([0.7, 0.0, 1.9], device=DEV)
    lines = sp.Lines.parallel(view, bins, -25.0, 0.5)
    plan = sp.Plan(sp.Grid(n, n, 0), lines)
    plan.set_paths(path, path)
    got = plan.fwd(torch.from_numpy(coef).to(DEV)).cpu().numpy().reshape(3, bins)
    # the line of direction (1, 0) with offset y = <P, (0, -1)> lies at x2 = -y
    W = np.array([_weights(25.0 - 0.5 * b, n) for b in range(bins)])
    assert np.array_equal(got[1], W @ coef.sum(1))
    p = np.zeros((3, bins), dtype=np.float32)
    p[1] = rng.integers(-8, 9, bins)
    back = plan.adj(torch.from_numpy(p.ravel()).to(DEV)).cpu().numpy()
    assert np.array_equal(back, np.repeat((p[1] @ W)[:, None], n, 1))
    plan.close()
