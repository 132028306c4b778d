"""Device memory that the training calls take, against what include/nrv.h states."""
import pytest

from gpu_util import make_params, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,pixel_bytes", [(1, 358), (0, 716)])
def test_backward_workspace(prec, pixel_bytes):
    """The first backward at 16 x 256 x 256 (BF16) and 2 x 256 x 256 (FP32): gradient tensors of
    pixel_bytes a canvas pixel and at most 128 MB of partial sums (2 MB more for the rounding of
    each of the two allocations)."""
    import torch
    from paper_2407_19097_gb300 import nrv
    c0, n, h, w = 5, 16 if prec == 1 else 2, 256, 256
    dev = torch_dev()
    net = nrv.Net(c0)
    p = torch.from_numpy(make_params(c0, seed=1)).to(dev)
    net.set_params(p)
    x = torch.zeros((n, h, w, 8), dtype=torch.bfloat16 if prec == 1 else torch.float32, device=dev)
    x[..., :c0] = 0.5
    rgb = torch.empty((n, h, w, 3), device=dev)
    d, g = torch.ones_like(rgb), torch.empty_like(p)
    warm = nrv.Net(c0)                     # kernels loaded, streams made
    warm.set_params(p)
    warm.forward_train(x, n, h, w, prec, rgb)
    warm.backward(d, g)
    net.forward_train(x, n, h, w, prec, rgb)
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info(dev)
    net.backward(d, g)
    torch.cuda.synchronize()
    took = free0 - torch.cuda.mem_get_info(dev)[0]
    print(f"prec {prec}: {took / 1e6:.1f} MB")
    assert took <= pixel_bytes * n * h * w + 128e6 + (4 << 20)
