"""FP32 results do not depend on how many images share a call: images and views computed together
equal, bit for bit, the same ones computed one at a time.  Sizes at which the deep levels of one
image leave most of the chip idle, so that any choice made from the whole batch would differ."""
import numpy as np
import pytest

import nrv_inputs as I
from gpu_util import make_params, torch_dev, upload_scene
from oracle import unet

pytestmark = pytest.mark.gpu
C0 = 5
NAMES = [l[0] for l in unet.layers(C0)]


def _net(seed=3):
    import torch
    from paper_2407_19097_gb300 import nrv
    net = nrv.Net(C0)
    net.set_params(torch.from_numpy(make_params(C0, seed=seed, bias_sigma=0.1)).to(torch_dev()))
    return net


@pytest.mark.parametrize("n,h,w", [(4, 512, 512), (3, 544, 960), (5, 256, 256), (16, 64, 64), (7, 40, 72)])
def test_shade_f32(n, h, w):
    import torch
    from paper_2407_19097_gb300 import nrv
    net, dev = _net(), torch_dev()
    x = torch.zeros((n, h, w, 8), device=dev)
    x[..., :C0] = torch.randn((n, h, w, C0), device=dev, generator=torch.Generator(device=dev).manual_seed(h))
    y, one = torch.empty((n, h, w, 3), device=dev), torch.empty((1, h, w, 3), device=dev)
    net.shade(x, n, h, w, nrv.PREC_F32, y)
    for i in range(n):
        net.shade(x[i:i + 1], 1, h, w, nrv.PREC_F32, one)
        assert torch.equal(y[i], one[0]), i


@pytest.mark.parametrize("n", [2, 6])
@pytest.mark.parametrize("name", ["e1b", "e2b", "e3a", "e3b", "up3", "d2a", "up2", "d1a", "up1", "d0a"])
def test_data_gradients_f32(name, n):
    """Each layer at its level of a 256 x 256 image."""
    import torch
    from paper_2407_19097_gb300 import nrv
    net, dev = _net(), torch_dev()
    layer = NAMES.index(name)
    _, kind, ci, co = unet.layers(C0)[layer]
    up = 2 if kind == "convT2" else 1
    size = 256 >> {"0": 0, "1": 1, "2": 2, "3": 3}[name[2] if up == 2 else name[1]]
    g = torch.Generator(device=dev).manual_seed(layer)
    dy = torch.randn((n, up * size, up * size, co), device=dev, generator=g)
    mask = torch.randn((n, size, size, ci), device=dev, generator=g)
    dx, one = torch.empty_like(mask), torch.empty_like(mask[:1])
    net.layer_dgrad(layer, dy, mask, n, size, size, nrv.PREC_F32, dx)
    for i in range(n):
        net.layer_dgrad(layer, dy[i:i + 1], mask[i:i + 1], 1, size, size, nrv.PREC_F32, one)
        assert torch.equal(dx[i], one[0]), i


def test_grouped_views_f32():
    """Four 512 x 512 views, shaded by one network call in a batch."""
    import torch
    from paper_2407_19097_gb300 import nrv
    sc = I.terrain_scene(300, seed=7)
    c0 = len(sc.channels) + 2
    scene, dev = upload_scene(sc), torch_dev()
    net = nrv.Net(c0)
    net.set_params(torch.from_numpy(make_params(c0, seed=8, bias_sigma=0.05)).to(dev))
    views = I.orbit_views(sc, [(512, 512)] * 4, seed=3)
    ds, do = I.depth_normalisation(sc, views[0])
    desc = nrv.make_pack_desc(sc.channels, ds, do)
    outs = [torch.empty((512, 512, 3), device=dev) for _ in views]
    one = torch.empty((512, 512, 3), device=dev)
    nrv.render_batch(scene, net, desc, views, outs, nrv.PREC_F32)
    for v, o in zip(views, outs):
        nrv.render_batch(scene, net, desc, [v], [one], nrv.PREC_F32)
        torch.cuda.synchronize()
        assert torch.equal(o, one)
