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
