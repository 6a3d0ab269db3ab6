"""Distinct views driven by distinct threads from a process's first frames on,
with blends of every kind: the images are those of one thread."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys, threading
sys.path.insert(0, %r)
import torch, scenegen, paper_2506_02774_gb300 as vgr
sc = scenegen.make_scene("tiny")
h = vgr.Hierarchy(sc)
kinds = [dict(), dict(), dict(tile_size=32), dict(tile_size=8), dict(blend_depth=48), dict(filter=vgr.FILTER_CANONICAL)]
cams = [scenegen.camera((-3.0 + 0.1 * k, 10.0, 2.5), 0.02 * k, 1283, 721, 700.0) for k in range(4)]
views = [vgr.View(h, **kw) for kw in kinds]
out, start = [None] * len(views), threading.Barrier(len(views))
def walk(i):
    torch.cuda.set_device(0)
    start.wait()
    out[i] = [views[i].render(c, 3.0).image().cpu() for c in cams]
threads = [threading.Thread(target=walk, args=(i,)) for i in range(len(views))]
[t.start() for t in threads]
[t.join() for t in threads]
for i, kw in enumerate(kinds):
    v = vgr.View(h, **kw)
    for c, img in zip(cams, out[i]):
        assert torch.equal(v.render(c, 3.0).image().cpu(), img), kw
print("threads ok")
""" % ROOT


def test_first_frames_on_several_threads():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=120, cwd=ROOT)
    assert r.returncode == 0 and "threads ok" in r.stdout, r.stderr[-2000:]
