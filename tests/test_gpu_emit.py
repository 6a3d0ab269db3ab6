"""The emission's pair list against the candidate rectangles it enumerates: in
the canonical mode every candidate tile of every visible Gaussian is a pair, so
the sorted list follows from the rectangles and the depth order alone.  A few
Gaussians that cover the whole image make chunks of slots that lie inside one
Gaussian, start or end in the middle of one, and end ragged."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402


def _scene(n, scale):
    leaves = scenegen.gen_leaves(n, 3, kind="box", sh_degree=0, box=(0.0, 30.0, 0.0, 30.0, 0.0, 8.0),
                                 logscale=(scale, 0.8))
    return scenegen.build_tree(leaves)


@pytest.mark.parametrize("n,scale", [(3, 2.0), (60, 1.5), (3000, -1.0), (30000, -3.0)])
@pytest.mark.parametrize("size,tile", [((640, 360), 8), ((333, 211), 16), ((1920, 1080), 32), ((8192, 4100), 8)])
def test_pairs_follow_the_rectangles(n, scale, size, tile):
    if n > 100 and size[0] > 2000:
        pytest.skip("one small case at the largest tile grid is enough")
    h = vgr.Hierarchy(_scene(n, scale))
    v = vgr.View(h, filter=vgr.FILTER_CANONICAL, tile_size=tile, use_graph=True)
    cam = scenegen.camera((-3.0, 15.0, 4.0), 0.0, size[0], size[1], 0.5 * size[0])
    for _ in range(2):
        r = v.render(cam, 0.0)
    d = v.debug()
    x0, y0 = d["vis_rect"][:, 0] & 0xFFFF, d["vis_rect"][:, 0] >> 16
    x1, y1 = d["vis_rect"][:, 1] & 0xFFFF, d["vis_rect"][:, 1] >> 16
    w = (x1 - x0 + 1).astype(np.int64)
    cnt = w * (y1 - y0 + 1)
    np.testing.assert_array_equal(cnt, d["vis_ntile"])
    order = d["depth_order"].astype(np.int64)
    own = np.repeat(np.arange(order.size), cnt[order])  # depth rank of each slot
    g = order[own]
    loc = np.arange(own.size) - np.repeat(np.cumsum(cnt[order]) - cnt[order], cnt[order])
    key = (y0[g] + loc // w[g]) * d["tiles"][0] + x0[g] + loc % w[g]
    at = np.argsort(key, kind="stable")
    assert r.stats["pair_count"] == r.stats["candidate_pairs"] == own.size > 0
    np.testing.assert_array_equal(d["pair_tile"], key[at])
    np.testing.assert_array_equal(d["pair_rank"], own[at])
    assert (d["pair_rowmask"] == 0xFF).all()
    start = np.searchsorted(key[at], np.arange(d["tile_range"].shape[0] + 1))
    some = start[1:] > start[:-1]
    np.testing.assert_array_equal(d["tile_range"][some], np.stack([start[:-1], start[1:]], 1)[some])
    v.close(); h.close()
