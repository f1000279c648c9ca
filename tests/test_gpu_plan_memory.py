"""A plan whose strip kernels' records no longer fit in device memory, but whose
line records and footprint tables do, runs on the general kernels."""
import math

import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("paper_2503_20907_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda"
MIB = 1 << 20


def test_a_plan_beside_a_nearly_full_device():
    n, m = 256, 2000000
    g = torch.Generator(DEV).manual_seed(3)
    a = torch.rand((2, m), device=DEV, generator=g) * (2.0 * math.pi)
    src = (0.75 * n * torch.stack([a[0].cos(), a[0].sin()], 1)).contiguous()
    dst = (0.75 * n * torch.stack([a[1].cos(), a[1].sin()], 1)).contiguous()
    grid, lines = sp.Grid(n, n, 3), sp.Lines.points(src, dst)
    coef, p = torch.rand((n, n), device=DEV, generator=g), torch.rand(m, device=DEV, generator=g)
    whole = sp.Plan(grid, lines)
    want = whole.fwd(coef), whole.adj(p)
    whole.set_paths(2, 2)
    general = whole.fwd(coef)
    whole.close()
    sino, back = torch.empty_like(p), torch.empty_like(coef)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # per line 64 bytes of record and 1,312 of table, then 208 and the order's 17:
    # room for the first two and 100 MiB
    room = m * (64 + 1312) + 100 * MIB
    free, total = torch.cuda.mem_get_info()
    if free < room + 1024 * MIB:
        pytest.skip("device memory in use elsewhere")
    hog = torch.empty(free - room, dtype=torch.uint8, device=DEV)
    try:
        left = torch.cuda.mem_get_info()[0]
        if not m * 1376 + 20 * MIB < left < m * 1584:
            pytest.skip("device memory in use elsewhere")
        plan = sp.Plan(grid, lines)
        plan.fwd(coef, sino)
        plan.adj(p, back)
        with pytest.raises(sp.SplineError):      # row records are the strip kernels'
            plan.set_records(True)
        torch.cuda.synchronize()
        plan.close()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(sino, general)
    # sums of at most 2^12 rounded terms per line, 2^21 atomic additions per node
    assert float((sino - want[0]).norm() / want[0].norm()) < 2e-6
    assert float((back - want[1]).norm() / want[1].norm()) < 1e-5
