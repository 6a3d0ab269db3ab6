"""The debug arrays of a view that lost its image buffers: a frame too large for
the memory that is left frees the old tile ranges and reports VGR_E_NOMEM.  The
records of the last frame are still there; what was lost stays out, and no kernel
reads it."""
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


def test_debug_after_a_lost_image(small_sh3_scene):
    h = vgr.Hierarchy(small_sh3_scene)
    v = vgr.View(h)
    cam = scenegen.camera((2.0, 15.0, 3.0), 0.2, 328, 250, 260.0)
    img = v.render(cam, 3.0).image().clone()
    before = v.debug()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
    with pytest.raises(vgr.VgrError) as e:  # 3.2 GB
        v.render(scenegen.camera((2.0, 15.0, 3.0), 0.2, 16384, 16384, 8000.0), 3.0)
    assert e.value.status == _abi.VGR_E_NOMEM
    d = _abi.DebugBuffers()
    _abi.check(_abi.load().vgr_view_debug(v.handle, ctypes.byref(d)))
    assert not d.tile_range and not d.pair_tile and d.n_pairs == before["n_pairs"]
    after = v.debug()
    for k in ("vis_node", "vis_depth", "vis_rect", "vis_recA", "vis_recB", "vis_rgb", "depth_order", "pair_rank"):
        np.testing.assert_array_equal(after[k], before[k])
    del hold
    torch.cuda.empty_cache()
    assert torch.equal(v.render(cam, 3.0).image(), img)
    again = v.debug()
    for k in ("tile_range", "pair_tile", "depth_order"):
        np.testing.assert_array_equal(again[k], before[k])
    v.close(); h.close()
