"""The whole-network calls (include/warmstart_conv.h, sp_convnet_*) behind
WarmStartNet against the FP64 oracle layers.  Weights, biases, images and
gradients are small integers, chosen so that every activation and every
gradient between layers is an integer of at most 256 in magnitude (exact in
BF16) and every sum is exact in FP32: results must equal the oracle's exactly,
whatever the order of the sums."""
import numpy as np
import pytest

from oracle.conv import conv3x3, conv3x3_grad_input, conv3x3_grad_weight

torch = pytest.importorskip("torch")
ws = pytest.importorskip("paper_2503_20907_gb300.warmstart")


def _case(B, H, W, seed):
    rng = np.random.default_rng(seed)
    params = []
    for cin, cout, _, _ in ws.LAYERS:
        w = np.zeros((cout, 9 * cin))
        if cout == 1:
            w[:] = rng.integers(-1, 2, w.shape)
        else:
            for o in range(cout):      # two taps per output keep the values small
                w[o, rng.choice(9 * cin, 2, replace=False)] = rng.choice([-1.0, 1.0], 2)
        params.append((w.reshape(cout, 3, 3, cin), rng.integers(-1, 2, cout).astype(np.float64)))
    return params, rng.integers(-2, 3, (B, H, W)).astype(np.float64), rng.integers(-1, 2, (B, H, W)).astype(np.float64)


def _oracle(params, z, g):
    """x_0, dz and the gradients of weights and biases."""
    xs = [z[..., None]]
    for (w, b), (_, _, relu, d) in zip(params, ws.LAYERS):
        y = conv3x3(xs[-1], w, b, d=d)
        xs.append(np.maximum(y, 0) if relu else y)
    gr, dws, dbs = g[..., None], [], []
    for k in reversed(range(len(params))):
        if ws.LAYERS[k][2]:
            gr = gr * (xs[k + 1] > 0)
        dw, db = conv3x3_grad_weight(xs[k], gr, d=ws.LAYERS[k][3])
        dws.append(dw), dbs.append(db)
        gr = conv3x3_grad_input(gr, params[k][0], d=ws.LAYERS[k][3])
        assert np.abs(gr).max() <= 256 and np.abs(dw).max() < 2 ** 23
    assert max(np.abs(x).max() for x in xs[:-1]) <= 256
    return z + xs[-1][..., 0], g + gr[..., 0], dws[::-1], dbs[::-1]


SIZES = [(1, 1, 1), (1, 3, 130), (2, 40, 33), (1, 37, 257), (3, 17, 128)]


def test_the_inputs_are_exact():
    for s in SIZES:
        _oracle(*_case(*s, seed=sum(s)))


def _net(params):
    net = ws.WarmStartNet()
    with torch.no_grad():
        for k, (w, b) in enumerate(params):
            net.w[k].copy_(torch.from_numpy(w))
            net.b[k].copy_(torch.from_numpy(b))
    return net.cuda()


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,W", SIZES)
def test_network_equals_the_oracle(B, H, W):
    params, z, g = _case(B, H, W, seed=B + H + W)
    x0, dz, dws, dbs = _oracle(params, z, g)
    net = _net(params)
    zt = torch.from_numpy(z).float().cuda().requires_grad_(True)
    gt = torch.from_numpy(g).float().cuda()
    for form in ("plain", "strided"):     # strided: z and the gradient are not contiguous
        zi = zt if form == "plain" else zt.transpose(1, 2).contiguous().transpose(1, 2)
        gi = gt if form == "plain" else gt.transpose(1, 2).contiguous().transpose(1, 2)
        net.zero_grad()
        zt.grad = None
        y = net(zi)
        y.backward(gi)
        assert np.array_equal(y.detach().cpu().numpy(), x0), form
        assert np.array_equal(zt.grad.cpu().numpy(), dz), form
        for k in range(len(params)):
            assert np.array_equal(net.w[k].grad.cpu().numpy(), dws[k]), (form, k)
            assert np.array_equal(net.b[k].grad.cpu().numpy(), dbs[k]), (form, k)
    with torch.no_grad():                 # two slabs of activations instead of all
        assert np.array_equal(net(zt).cpu().numpy(), x0)


@pytest.mark.gpu
def test_network_forms():
    params, z, g = _case(2, 9, 20, seed=3)
    x0, _, dws, _ = _oracle(params, z, g)
    net = _net(params)
    zt, gt = torch.from_numpy(z).float().cuda(), torch.from_numpy(g).float().cuda()
    # inputs and weights changed between the passes: the backward is of the values that were used
    y = net(zt)
    zt.zero_()
    with torch.no_grad():
        net.w[1].mul_(2)
    y.backward(gt)
    assert np.array_equal(net.w[0].grad.cpu().numpy(), dws[0])
    # layer by layer (FP64 image) and under a captured graph
    net = _net(params)
    zt = torch.from_numpy(z).cuda()
    with torch.no_grad():
        assert np.array_equal(net(zt).cpu().numpy(), x0)
        zf, graph = zt.float(), torch.cuda.CUDAGraph()
        net(zf)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            y = net(zf)
        zf.zero_()
        graph.replay()
        zero = y.clone()
        zf.copy_(zt)
        graph.replay()
        assert np.array_equal(y.cpu().numpy(), x0) and not torch.equal(zero, y)
