"""Frames with 2^32 candidate slots or more: every Gaussian covers an image of
2^20 tiles.  Their 32-bit slot offsets wrap, so the emission has to leave them
alone; the frame is refused as documented, by the partition and by the radix
passes with the slot scan, and the view renders the next frame as a new one
does."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402
from paper_2506_02774_gb300 import _abi  # noqa: E402

RADIX_DEPTH = 4  # VGR_HOOK_RADIX_DEPTH


def _wide_leaves(n):
    """n Gaussians of 200 m standard deviation around (10, 0, 0)."""
    leaves = scenegen.gen_leaves(n, 5, kind="box", sh_degree=0, box=(9.0, 11.0, -1.0, 1.0, -1.0, 1.0))
    leaves["cov6"] = np.tile(np.float32([4e4, 0, 0, 4e4, 0, 4e4]), (n, 1))
    leaves["opacity"] = np.full(n, 0.9, np.float32)
    leaves["rad2"] = scenegen.leaf_rad2(np.full((n, 3), 200.0))
    return scenegen.build_tree(leaves)


@pytest.mark.parametrize("hooks", [0, RADIX_DEPTH])
@pytest.mark.parametrize("n", [4096, 4097, 8192])  # 2^32 slots, 2^32 and 2^20 more, 2^33
def test_frame_is_refused(n, hooks):
    h = vgr.Hierarchy(_wide_leaves(n))
    v, new = vgr.View(h, tile_size=8, test_hooks=hooks), vgr.View(h, tile_size=8)
    with pytest.raises(vgr.VgrError) as e:
        v.render(scenegen.camera((0.0, 0.0, 0.0), 0.0, 8192, 8192, 4000.0), 0.0)
    assert e.value.status == _abi.VGR_E_OVERFLOW
    small = scenegen.camera((0.0, 0.0, 0.0), 0.0, 48, 40, 24.0)
    a, b = v.render(small, 0.0), new.render(small, 0.0)
    assert a.stats["visible_count"] == b.stats["visible_count"] == n
    assert a.stats["candidate_pairs"] == b.stats["candidate_pairs"] == n * 30
    assert torch.equal(a.image(), b.image())
    v.close(); new.close(); h.close()
