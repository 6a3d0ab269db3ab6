"""The debug view's depth order holds every entry in front of the camera, as the
header has it: the visible ones by (depth key, index), then the culled ones,
ascending -- from the partition as from the radix passes, on a second frame with
fewer visible entries too; and the culled entries' records are zeros."""
import ctypes

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402
from paper_2506_02774_gb300 import _abi  # noqa: E402


def _u32(ptr, n):
    return vgr.device_tensor(ptr, (n,), "int32").cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("hooks", [0, 4])  # VGR_HOOK_RADIX_DEPTH
@pytest.mark.parametrize("n", [1, 900, 30000])
def test_whole_order(n, hooks):
    leaves = scenegen.gen_leaves(n, 3, kind="box", sh_degree=0, box=(0.0, 30.0, 0.0, 30.0, 0.0, 8.0), logscale=(-3.0, 0.5))
    leaves["opacity"] = leaves["opacity"].copy()
    leaves["opacity"][::3] = 0.001  # below alpha*: culled after the cut
    h = vgr.Hierarchy(scenegen.build_tree(leaves))
    v = vgr.View(h, test_hooks=hooks)
    for yaw in (0.0, 0.6):
        r = v.render(scenegen.camera((-5.0, 15.0, 4.0), yaw, 333, 211, 160.0), 0.0)
        d = _abi.DebugBuffers()
        _abi.check(_abi.load().vgr_view_debug(v.handle, ctypes.byref(d)))
        nf, nv = int(d.n_front), int(d.n_visible)
        assert nf == r.stats["front_count"] and nv < nf
        if nf == 0:
            continue
        key, cnt, order = _u32(d.vis_depth, nf), _u32(d.vis_ntile, nf), _u32(d.depth_order, nf)
        np.testing.assert_array_equal(order, np.lexsort((np.arange(nf), key)))
        assert (cnt[order[:nv]] > 0).all() and (cnt[order[nv:]] == 0).all()
        for ptr, w in ((d.vis_rect, 2), (d.vis_recA, 4), (d.vis_recB, 4), (d.vis_rgb, 4)):
            rec = _u32(ptr, w * nf).reshape(nf, w)
            assert (rec[cnt == 0] == 0).all()
    v.close(); h.close()
