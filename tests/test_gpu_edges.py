"""The kernels of the network and of the render pass at the sizes where their tiles, splits and
vector loads end: one pixel, one past a tile, narrow levels, odd offsets, extreme depths.

A sum of K products in any order has an error of at most K u / (1 - K u) * sum |terms| (u = 2^-24),
the bound of the FP32 layers here; gradients also allow 1e-5 * sum |terms|, the bound of
test_gpu_layer_grad for the same sums."""
import numpy as np
import pytest

import nrv_inputs as I
import oracle
from gpu_util import make_params, psnr_range, torch_dev, upload_scene
from oracle import unet
from test_gpu_conv import _run
from test_gpu_layer_grad import C0, _bf16, _offsets
from test_gpu_raster import _every_variant

pytestmark = pytest.mark.gpu

NAMES = [l[0] for l in unet.layers(C0)]


def _gamma(k):
    return k * 2.0 ** -24 / (1 - k * 2.0 ** -24)


def _net(seed):
    import torch
    from paper_2407_19097_gb300 import nrv
    flat = make_params(C0, seed=seed, bias_sigma=0.1)
    net = nrv.Net(C0)
    net.set_params(torch.from_numpy(flat).to(torch_dev()))
    return net, flat


# one pixel; past a 32- and a 64-pixel tile; 8, 16 and 32 rows plus one; several clusters per layer;
# a grid that fills the SMs without a split (the last)
SIZES = [(1, 1, 1), (1, 9, 33), (3, 17, 66), (2, 33, 31), (1, 130, 290)]


@pytest.mark.parametrize("n,h,w", SIZES)
@pytest.mark.parametrize("name", ["e0a", "e1b", "e3b", "d0a", "up3", "up1"])
def test_f32_layers(name, n, h, w):
    """Forward and data gradient of a layer in FP32."""
    import torch
    layer = NAMES.index(name)
    _, kind, ci, co = unet.layers(C0)[layer]
    net, flat = _net(layer + 3)
    rng = np.random.default_rng(layer)
    cin = 8 if layer == 0 else ci
    x = rng.standard_normal((n, h, w, cin)).astype(np.float32)
    x[..., ci:] = 0.0
    W, b = unet.unflatten(flat.astype(np.float64), C0)[name]
    xt = torch.from_numpy(x).to(torch_dev())
    c1 = cin // 2 if name == "d0a" else cin
    up = 2 if kind == "convT2" else 1
    y = torch.empty((n, up * h, up * w, co), device=torch_dev())
    _run(net, layer, xt[..., :c1].contiguous(), xt[..., c1:].contiguous() if c1 < cin else None,
         n, h, w, 0, y)
    xr = x[..., :ci].astype(np.float64)
    f, K = (unet.conv3, 9 * ci) if kind == "conv3" else (unet.convT2, ci)
    ref = f(xr, W, b)
    if kind == "conv3":
        ref = unet.relu(ref)
    S = f(np.abs(xr), np.abs(W), np.abs(b))
    assert np.all(np.abs(y.cpu().numpy() - ref) <= _gamma(K + 1) * S)
    if layer == 0:
        return
    dy = rng.standard_normal((n, up * h, up * w, co)).astype(np.float32)
    dx = torch.empty((n, h, w, ci), device=torch_dev())
    mask = rng.standard_normal((n, h, w, ci)).astype(np.float32)
    net.layer_dgrad(layer, torch.from_numpy(dy).to(torch_dev()), torch.from_numpy(mask).to(torch_dev()),
                    n, h, w, 0, dx)
    bwd, K = (unet.conv3_bwd, 9 * co) if kind == "conv3" else (unet.convT2_bwd, 4 * co)
    zero = np.zeros((n, h, w, ci))
    ref = np.where(mask > 0, bwd(zero, W, dy.astype(np.float64))[0], 0.0)
    S = bwd(zero, np.abs(W), np.abs(dy).astype(np.float64))[0]
    assert np.all(np.abs(dx.cpu().numpy() - ref) <= _gamma(K) * S)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (1, 9, 32), (2, 5, 33), (2, 8, 64), (3, 3, 65), (1, 20, 129)])
@pytest.mark.parametrize("name", ["e0b", "e2a", "d2a", "e3b", "up2"])
def test_weight_gradient_tiles(name, n, h, w, prec):
    """Weight gradients over images narrower and wider than each tile width."""
    import torch
    layer = NAMES.index(name)
    _, kind, ci, co = unet.layers(C0)[layer]
    net, _ = _net(1)
    rng = np.random.default_rng(layer)
    up = 2 if kind == "convT2" else 1
    x = rng.standard_normal((n, h, w, ci)).astype(np.float32)
    dy = rng.standard_normal((n, up * h, up * w, co)).astype(np.float32)
    if prec == 1:
        x, dy = _bf16(x).astype(np.float32), _bf16(dy).astype(np.float32)
    dt = torch.bfloat16 if prec == 1 else torch.float32
    xt, dyt = (torch.from_numpy(a).to(torch_dev()).to(dt) for a in (x, dy))
    c1 = ci // 2 if name == "d2a" else ci
    off, total = _offsets(C0)
    grad = torch.full((total,), float("nan"), device=torch_dev())
    net.layer_wgrad(layer, dyt, xt[..., :c1].contiguous(), xt[..., c1:].contiguous() if c1 < ci else None,
                    n, h, w, prec, grad)
    g = grad.cpu().numpy().astype(np.float64)
    bwd = unet.conv3_bwd if kind == "conv3" else unet.convT2_bwd
    x, dy = x.astype(np.float64), dy.astype(np.float64)
    wz = np.zeros(unet.weight_shape(kind, ci, co))
    _, dw, db = bwd(x, wz, dy)
    _, dw_abs, db_abs = bwd(np.abs(x), wz, np.abs(dy))
    o, wsz, ob, _ = off[name]
    rel = max(1e-5, _gamma(up * up * n * h * w))
    assert np.all(np.abs(g[o:o + wsz].reshape(dw.shape) - dw) <= rel * dw_abs + 1e-30)
    assert np.all(np.abs(g[ob:ob + co] - db) <= rel * db_abs + 1e-30)
    assert np.all(np.isnan(np.concatenate([g[:o], g[ob + co:]])))


@pytest.mark.parametrize("prec", [0, 1])
def test_backward_captured_on_a_side_stream(prec):
    """The backward pass runs weight gradients beside data gradients on a stream of its own: in a
    captured graph, replayed with other contents, it makes the gradients of the eager call."""
    import torch
    n, h, w = 2, 24, 40
    net, flat = _net(2)
    rng = np.random.default_rng(4)
    dev = torch_dev()
    dt = torch.bfloat16 if prec == 1 else torch.float32
    x = torch.zeros((n, h, w, 8), dtype=dt, device=dev)
    x[..., :C0] = torch.from_numpy(rng.standard_normal((n, h, w, C0))).to(dt)
    d = torch.from_numpy(rng.standard_normal((n, h, w, 3)).astype(np.float32)).to(dev)
    rgb = torch.empty((n, h, w, 3), device=dev)
    grad = torch.zeros(flat.size, device=dev)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        net.forward_train(x, n, h, w, prec, rgb)
        net.backward(d, grad)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        net.forward_train(x, n, h, w, prec, rgb)
        net.backward(d, grad)
    x[..., :C0] *= -0.5
    d.mul_(2.0)
    graph.replay()
    torch.cuda.synchronize()
    got = grad.clone()
    net.forward_train(x, n, h, w, prec, rgb)
    net.backward(d, grad)
    torch.cuda.synchronize()
    assert torch.equal(got, grad) and float(got.abs().max()) > 0


@pytest.mark.parametrize("h,w", [(24, 264), (56, 40)])
def test_fp8_network_ragged(h, w):
    """Levels whose widths are no multiple of a tile, through the pools, encoders and decoders
    fused into the FP8 layers; the accuracy bar of the weaker all-E4M3 mode of test_gpu_fp8."""
    import torch
    from paper_2407_19097_gb300 import nrv
    net, flat = _net(5)
    dev = torch_dev()
    rng = np.random.default_rng(h)
    x = np.zeros((2, h, w, 8), np.float32)
    x[..., :C0] = _bf16(rng.standard_normal((2, h, w, C0)))
    xb = torch.from_numpy(x).to(dev).to(torch.bfloat16)
    net.calibrate(xb, 2, h, w)
    out = torch.empty((2, h, w, 3), device=dev)
    net.shade(xb, 2, h, w, nrv.PREC_FP8, out)
    ref = unet.forward(x[..., :C0].astype(np.float64), unet.unflatten(flat, C0))
    got = out.cpu().numpy()
    p, err = psnr_range(got, ref), float(np.abs(got - ref).max())
    assert p >= 40.0 and err <= 0.15, (p, err)


@pytest.mark.parametrize("off", [(0, 0, 0), (1, 1, 1), (0, 2, 0), (0, 0, 3)])
@pytest.mark.parametrize("n", [1, 3, 1027, 400_001])
def test_l1_offsets(n, off):
    """Buffers that start off a 16-byte boundary, each on its own."""
    import torch
    from paper_2407_19097_gb300 import nrv
    rng = np.random.default_rng(n)
    y, t = rng.standard_normal((2, n)).astype(np.float32)
    t[::5] = y[::5]
    bufs = [torch.empty(n + 4, device=torch_dev())[o:o + n] for o in off]
    bufs[0].copy_(torch.from_numpy(y))
    bufs[1].copy_(torch.from_numpy(t))
    loss = torch.zeros(1, device=torch_dev())
    nrv.l1_loss(bufs[0], bufs[1], loss, bufs[2])
    diff = y - t
    ref = np.abs(diff).astype(np.float64).mean()
    assert abs(loss.item() - ref) <= _gamma(n + 2) * ref
    assert np.array_equal(bufs[2].cpu().numpy(), np.sign(diff) * np.float32(1.0 / np.float32(n)))


def test_depths_beyond_the_fast_range(simple_view):
    """Depths from 1e-30 to 1e30 (the corrected quotient covers 2^-60 .. 2^125 only), one view and
    three of unequal size and range, every variant, bit for bit."""
    rng = np.random.default_rng(9)
    z = (10.0 ** rng.uniform(-30, 30, 5003)).astype(np.float32)
    u = rng.uniform(-0.6, 0.6, (5003, 2)).astype(np.float32)
    pts = np.ascontiguousarray(np.concatenate([u * z[:, None], z[:, None]], 1).astype(np.float32))
    sc = I.Scene("depths", pts, np.arange(4 * 5003, dtype=np.uint32).reshape(-1, 4), 4, [])
    m = [2, 0, 0, 0, 0, 2, 0, 0, 0, 0, 0, 0, 0, 0, 1, 0]
    views = [simple_view(m, 300, 200, 1e-30, 3e38), simple_view(m, 65, 33, 1e-3, 1e3),
             simple_view(m, 17, 300, 1e-25, float("inf"))]
    upload_scene(sc)
    refs = _every_variant(sc, views[:1])
    assert (refs[0][2] > 0).mean() > 0.05
    _every_variant(sc, views)
