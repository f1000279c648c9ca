"""Sequences of plan and batch calls in which what one call leaves behind
decides what another gives: graphs with a captured prepare that are replayed
with other angles, and empty line lists."""
import pytest

import workloads

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _case(degree=3, n=48, bins=70):
    view = torch.linspace(0.0, 3.0, 31, device=DEV)
    grid, lines = sp.Grid(n, n, degree, 1.0), sp.Lines.parallel(view, bins, -0.5 * (bins - 1), 1.0)
    coef = torch.from_numpy(workloads.ellipse_phantom(n, 8, 4, radius=n / 3, axes=(2.0, n / 5))).to(DEV)
    p = torch.rand(lines.m, device=DEV, generator=torch.Generator(DEV).manual_seed(1)) - 0.3
    return view, grid, lines, coef, p


def _close(a, b):
    # the same kernels on the same line data: only the order of the adjoints'
    # atomic additions differs
    return float((a - b).norm() / b.norm()) < 2e-6


def _fresh(grid, lines, coef, p, paths):
    plan = sp.Plan(grid, lines)
    plan.set_paths(*paths)
    out = plan.fwd(coef), plan.adj(p)
    plan.close()
    return out


def _capture(f):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        f()
    return graph


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("paths", [(2, 2), (2, 3)])
@pytest.mark.parametrize("warm", [False, True])
def test_projections_after_a_replayed_prepare(paths, warm, degree):
    # the prepare is captured on the strip kernels' path (no footprint tables)
    # and replayed when the plan has gone over to kernels that read them
    view, grid, lines, coef, p = _case(degree)
    plan = sp.Plan(grid, lines, prepare=warm)
    graph = _capture(plan.prepare)
    graph.replay()
    plan.set_paths(*paths)
    first = plan.fwd(coef)
    want = _fresh(grid, lines, coef, p, paths)
    assert torch.equal(first, want[0]) and _close(plan.adj(p), want[1])
    for _ in range(2):
        view.add_(0.21)
        graph.replay()
        want = _fresh(grid, lines, coef, p, paths)
        assert not _close(first, want[0])
        for _ in range(2):               # (each builds the tables again)
            assert torch.equal(plan.fwd(coef), want[0]) and _close(plan.adj(p), want[1])
    plan.prepare()                       # and an ordinary prepare again
    assert torch.equal(plan.fwd(coef), want[0]) and _close(plan.adj(p), want[1])
    plan.close()


@pytest.mark.parametrize("degree", [0, 2, 3])
@pytest.mark.parametrize("paths", [(0, 0), (2, 2), (2, 3)])
def test_a_graph_of_prepare_and_projections(paths, degree):
    view, grid, lines, coef, p = _case(degree)
    plan = sp.Plan(grid, lines)
    plan.set_paths(*paths)
    sino, back = torch.empty(lines.m, device=DEV), torch.empty(grid.ny, grid.nx, device=DEV)
    plan.fwd(coef, sino)

    def step():
        plan.prepare()
        plan.fwd(coef, sino)
        plan.adj(p, back)

    graph = _capture(step)
    for _ in range(2):
        view.add_(0.21)
        graph.replay()
        want = _fresh(grid, lines, coef, p, paths)
        assert torch.equal(sino, want[0]) and _close(back, want[1])
        # eager projections of the plan that the graph prepared
        assert torch.equal(plan.fwd(coef), want[0]) and _close(plan.adj(p), want[1])
    plan.close()


@pytest.mark.parametrize("degree,basis", [(1, 0), (2, 0), (3, 0), (1, 1)])
def test_a_captured_projection_replayed(degree, basis):
    # captured before any projection of its path has run: the graph builds the
    # tables, at every replay
    view, _, lines, coef, p = _case(degree)
    grid = sp.Grid(coef.shape[1], coef.shape[0], degree, 1.0, basis=basis)
    want = _fresh(grid, lines, coef, p, (2, 2))
    plan = sp.Plan(grid, lines)
    plan.set_paths(2, 2)
    sino = torch.empty(lines.m, device=DEV)
    graph = _capture(lambda: plan.fwd(coef, sino))
    for _ in range(3):
        sino.zero_()
        graph.replay()
        assert torch.equal(sino, want[0])
        assert torch.equal(plan.fwd(coef), want[0]) and _close(plan.adj(p), want[1])
    plan.close()


@pytest.mark.parametrize("paths", [(0, 0), (1, 1), (2, 2)])
@pytest.mark.parametrize("degree", [0, 3])
def test_empty_line_lists(degree, paths):
    view, grid, lines, coef, p = _case(degree)
    none = sp.Lines.theta_y(torch.empty(0, device=DEV), torch.empty(0, device=DEV))
    plan = sp.Plan(grid, none)
    plan.set_paths(*paths)
    empty = torch.empty(0, device=DEV)
    assert plan.fwd(coef).numel() == 0
    assert torch.equal(plan.adj(empty, torch.full_like(coef, 7.0)), torch.zeros_like(coef))
    x, gamma = plan.cgls(empty, 2, x0=coef)
    assert torch.equal(x, coef) and not gamma.any()
    plan.close()


@pytest.mark.parametrize("degree", [0, 3])
def test_a_batch_with_an_empty_line_list(degree):
    view, grid, lines, coef, p = _case(degree)
    none = sp.Lines.points(torch.empty(0, 2, device=DEV), torch.empty(0, 2, device=DEV))
    empty = torch.empty(0, device=DEV)
    batch = sp.Batch([grid, grid, grid], [lines, none, lines])
    want = _fresh(grid, lines, coef, p, (0, 0))
    out = batch.fwd([coef] * 3)
    back = batch.adj([p, empty, p], [torch.full_like(coef, 7.0) for _ in range(3)])
    assert torch.equal(out[0], want[0]) and out[1].numel() == 0 and torch.equal(out[2], want[0])
    assert _close(back[0], want[1]) and _close(back[2], want[1])
    assert torch.equal(back[1], torch.zeros_like(coef))
    batch.close()
