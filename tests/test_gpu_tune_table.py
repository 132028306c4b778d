"""A render-pass choice belongs to the table of variants it was made from: a saved file of another
table selects nothing."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

SCRIPT = r'''
import sys
sys.path.insert(0, {root!r})
import torch
import nrv_inputs as I
from paper_2407_19097_gb300 import nrv
from gpu_util import upload_scene
sc = I.cube_scene(1_100_000, k=3, seed=2)               # the render pass tunes from 2^20 points on
scene = upload_scene(sc)
keys = [torch.empty((96, 128), dtype=torch.int64, device="cuda:0") for _ in range(2)]
views = [I.cube_view(128, 96) for _ in keys]
nrv.rasterize(scene, views[:1], keys[:1])
nrv.rasterize(scene, views, keys)
torch.cuda.synchronize()
nrv.tune_save(sys.argv[1])
print("timings", nrv.lib().nrv_tune_timings())
'''


def _run(tmp, cache, out):
    script = tmp / "run.py"
    script.write_text(SCRIPT.format(root=ROOT))
    env = dict(os.environ, PYTHONPATH=os.path.join(ROOT, "tests"), NRV_TUNE_CACHE=str(cache))
    env.pop("NRV_VIS_VARIANT", None)
    r = subprocess.run([sys.executable, str(script), str(out)], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return int([l for l in r.stdout.splitlines() if l.startswith("timings")][-1].split()[1])


def test_choices_of_another_table_are_timed_again(tmp_path):
    # as written before the variants were reordered
    old = tmp_path / "old.txt"
    old.write_text("render multi=0 log2n=20 = 3\nrender multi=1 log2n=20 = 2\n")
    saved = tmp_path / "new.txt"
    assert _run(tmp_path, old, saved) == 2
    assert _run(tmp_path, saved, tmp_path / "again.txt") == 0
    # the same lines with another table named are not taken either
    other = tmp_path / "other.txt"
    lines = [l for l in saved.read_text().splitlines() if l.startswith("render") and "table=" in l]
    assert len(lines) == 2
    other.write_text("\n".join(l.split("table=")[0] + "table=00000000 = 1" for l in lines) + "\n")
    assert _run(tmp_path, other, tmp_path / "third.txt") == 2
