"""Views with an unbounded far plane (or a near plane below 2^-60) cost what bounded ones do: the
plain division is for the points whose depth lies out there, not for every point.  Their keys are
checked against the oracle, every variant, in test_gpu_edges."""
import copy

import pytest

import nrv_inputs as I
from gpu_util import torch_dev, upload_scene

pytestmark = pytest.mark.gpu


def test_unbounded_far_plane_keeps_its_speed(monkeypatch):
    """The first variant over 9M points and eight views; the fastest of 40 alternating passes each
    (1.05 times the bounded views, and 1.30 with every point divided again)."""
    import torch
    from paper_2407_19097_gb300 import nrv
    monkeypatch.setenv("NRV_VIS_VARIANT", "0")
    sc = I.terrain_scene(3000, seed=7)
    scene = upload_scene(sc)
    plain = I.orbit_views(sc, [(960, 540)] * 8, seed=3)
    wide = [copy.copy(v) for v in plain]
    for v in wide:
        v.zfar = float("inf")
    keys = [[torch.empty((540, 960), dtype=torch.int64, device=torch_dev()) for _ in plain] for _ in range(2)]
    best = [float("inf")] * 2
    for _ in range(40):
        for k, views in enumerate((plain, wide)):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            nrv.rasterize(scene, views, keys[k])
            b.record()
            b.synchronize()
            best[k] = min(best[k], a.elapsed_time(b))
    print(f"bounded {1e3 * best[0]:.1f} us, unbounded {1e3 * best[1]:.1f} us")
    assert all(torch.equal(a, b) for a, b in zip(*keys))
    assert best[1] <= 1.18 * best[0]
