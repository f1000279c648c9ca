"""A NaN pixel gives NaN wherever a tap sees it and nowhere else, through the
ReLUs too: single layers, and the network's receptive field."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
ws = pytest.importorskip("paper_2503_20907_gb300.warmstart")

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _spread(mask, d):
    """Pixels that see a marked pixel through a 3x3 stencil of spacing d."""
    out = np.zeros_like(mask)
    H, W = mask.shape
    for dy in (-d, 0, d):
        for dx in (-d, 0, d):
            y0, y1, x0, x1 = max(0, -dy), min(H, H - dy), max(0, -dx), min(W, W - dx)
            if y1 > y0 and x1 > x0:
                out[y0:y1, x0:x1] |= mask[y0 + dy:y1 + dy, x0 + dx:x1 + dx]
    return out


@pytest.mark.parametrize("relu", [False, True])
@pytest.mark.parametrize("cin,cout,d", [(1, 32, 1), (1, 32, 3), (32, 32, 1), (32, 32, 5), (32, 1, 1), (32, 1, 2)])
def test_a_layer(cin, cout, d, relu):
    H, W = 11, 140
    g = torch.Generator(DEV).manual_seed(cin + cout + d)
    x = torch.randn((1, H, W, cin), device=DEV, generator=g).bfloat16()
    w = torch.randn((cout, 3, 3, cin), device=DEV, generator=g) * 0.2
    b = torch.randn(cout, device=DEV, generator=g)
    mask = np.zeros((H, W), dtype=bool)
    for j, i in ((5, 40), (0, 0), (7, 129)):
        mask[j, i] = True
        x[0, j, i, cin // 2] = float("nan")
    y = ws.conv3x3(x, w, b, relu, d).float().reshape(H, W, cout).cpu().numpy()
    want = _spread(mask, d)
    assert np.isnan(y[want]).all() and np.isfinite(y[~want]).all()


def test_the_network():
    net, _ = ws.load_net(ws.DEFAULT_WEIGHTS, DEV)
    H, W = 150, 170
    z = torch.rand((2, H, W), device=DEV, generator=torch.Generator(DEV).manual_seed(4))
    with torch.no_grad():
        clean = net(z)
        z[1, 70, 90] = float("nan")
        want = np.zeros((H, W), dtype=bool)
        want[70, 90] = True
        for _, _, _, d in ws.LAYERS:
            want = _spread(want, d)
        y = net(z)
    assert torch.equal(y[0], clean[0])
    got = y[1].cpu().numpy()
    assert 100 < want.sum() < H * W and np.isnan(got[want]).all()
    assert np.array_equal(got[~want], clean[1].cpu().numpy()[~want])
