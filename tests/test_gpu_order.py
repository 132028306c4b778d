"""Calls that follow one another on a stream without a wait between them: what one call writes
is what the next one reads."""
import numpy as np
import pytest

from gpu_util import make_params, torch_dev

pytestmark = pytest.mark.gpu


def _input(n, h, w, c0, seed):
    import torch
    rng = np.random.default_rng(seed)
    x = torch.zeros((n, h, w, 8), dtype=torch.bfloat16, device=torch_dev())
    x[..., :c0] = torch.from_numpy(rng.standard_normal((n, h, w, c0))).to(torch.bfloat16)
    return x


def test_shade_reads_the_weights_just_set():
    """The first conv of a BF16 forward loads its weights ahead of its dependency wait: with new
    weights set immediately before, it must see those."""
    import torch
    from paper_2407_19097_gb300 import nrv
    c0, n, h, w = 5, 1, 64, 96
    dev = torch_dev()
    net = nrv.Net(c0)
    x = _input(n, h, w, c0, 1)
    flats = [torch.from_numpy(make_params(c0, seed=s, bias_sigma=0.1)).to(dev) for s in range(4)]
    refs = []
    for f in flats:
        net.set_params(f)
        torch.cuda.synchronize()
        y = torch.empty((n, h, w, 3), device=dev)
        net.shade(x, n, h, w, nrv.PREC_BF16, y)
        torch.cuda.synchronize()
        refs.append(y)
    outs = [torch.empty((n, h, w, 3), device=dev) for _ in range(200)]
    for i, y in enumerate(outs):
        net.set_params(flats[i % 4])
        net.shade(x, n, h, w, nrv.PREC_BF16, y)
    torch.cuda.synchronize()
    assert [i for i, y in enumerate(outs) if not torch.equal(y, refs[i % 4])] == []


def test_train_steps_back_to_back():
    """Each step's forward reads the weights that the step before it updated and packed: 40 steps
    in a row against the same steps with a wait after each."""
    import torch
    from paper_2407_19097_gb300 import nrv
    c0, n, h, w = 5, 2, 64, 64
    dev = torch_dev()
    x = _input(n, h, w, c0, 2)
    t = torch.rand((n, h, w, 3), device=dev, generator=torch.Generator(device=dev).manual_seed(3))

    def run(wait):
        net = nrv.Net(c0)
        p = torch.from_numpy(make_params(c0, seed=6, bias_sigma=0.1)).to(dev)
        net.set_params(p)
        g, m, v = (torch.zeros_like(p) for _ in range(3))
        losses = [torch.zeros(1, device=dev) for _ in range(40)]
        torch.cuda.synchronize()
        for i, loss in enumerate(losses):
            net.train_step(p, g, m, v, i + 1, 1e-2, x, t, n, h, w, nrv.PREC_BF16, loss)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return torch.cat(losses), p

    (la, pa), (lb, pb) = run(True), run(False)
    assert torch.equal(la, lb) and torch.equal(pa, pb)


@pytest.mark.parametrize("kind", ["l1", "recon"])
def test_losses_on_two_streams(kind):
    """Losses in flight on two streams at once, and a captured one replayed beside them, have
    partial sums of their own: each value is that of the call alone."""
    import torch
    from paper_2407_19097_gb300 import nrv
    dev = torch_dev()
    shapes = [(2, 512, 512, 3), (1, 64, 96, 3), (4, 512, 512, 3)]
    pairs = [[torch.rand(s, device=dev, generator=torch.Generator(device=dev).manual_seed(10 * i + j))
              for j in range(2)] for i, s in enumerate(shapes)]

    def call(i, out, d):
        y, t = pairs[i]
        if kind == "l1":
            nrv.l1_loss(y, t, out, d)
        else:
            nrv.recon_loss(y, t, (0.5, 1.0, 0.25), out, d)

    refs = []
    for i, (y, _) in enumerate(pairs):
        out, d = torch.zeros(1, device=dev), torch.empty_like(y)
        call(i, out, d)
        torch.cuda.synchronize()
        refs.append((out, d))
    streams = [torch.cuda.Stream() for _ in range(3)]
    rounds = 60
    outs = [torch.zeros((rounds, 1), device=dev) for _ in pairs]
    grads = [torch.empty_like(y) for y, _ in pairs]
    graph_out = torch.zeros(1, device=dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=streams[2]):
        call(2, graph_out, grads[2])
    torch.cuda.synchronize()
    for r in range(rounds):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                call(i, outs[i][r], grads[i])
        with torch.cuda.stream(streams[2]):
            graph.replay()
            outs[2][r].copy_(graph_out)
    torch.cuda.synchronize()
    for i, (ref, d) in enumerate(refs):
        assert torch.equal(outs[i], ref.expand(rounds, 1)), i
        assert torch.equal(grads[i], d), i


def test_views_that_share_planes():
    """One set of planes passed for all views of a call holds the last view's, as when the views are
    resolved one after the other."""
    import torch
    import nrv_inputs as I
    from gpu_util import gpu_raster, upload_scene
    from paper_2407_19097_gb300 import nrv
    sc = I.terrain_scene(300, seed=7)
    scene, dev = upload_scene(sc), torch_dev()
    views = I.orbit_views(sc, [(640, 480)] * 6, seed=3)
    k = scene.n_words
    keys = [torch.empty((480, 640), dtype=torch.int64, device=dev) for _ in views]
    depth = torch.empty((480, 640), dtype=torch.int32, device=dev)
    mask = torch.empty((480, 640), dtype=torch.uint8, device=dev)
    attr = torch.empty((k, 480, 640), dtype=torch.int32, device=dev)
    refs = gpu_raster(scene, views)
    assert not np.array_equal(refs[0][1], refs[-1][1])
    for _ in range(20):
        nrv.rasterize(scene, views, keys, [depth] * 6, [mask] * 6, [attr] * 6)
        torch.cuda.synchronize()
        for kt, ref in zip(keys, refs):
            assert np.array_equal(kt.cpu().numpy().view(np.uint64), ref[0])
        for t, ref in zip((depth, mask, attr), refs[-1][1:]):
            assert np.array_equal(t.cpu().numpy().view(ref.dtype), ref)
