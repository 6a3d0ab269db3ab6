"""Where a frame's route changes with its sizes: keys that just fit a depth bucket
and just do not, runs of equal depths around the ranking's limit, a single visible
Gaussian; frames around the one that tries the partition again after a bucket that
did not fit; a coarse cut from scratch in a tree with more than 2^24 nodes; host
images off a 16-byte boundary in the blend with two pixels per lane."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

RADIX_DEPTH, LOD_LEVELS = 4, 8  # VGR_HOOK_*


def _scene(n, depth):
    """n leaves, all in view of _cam, at x = depth(rng)."""
    leaves = scenegen.gen_leaves(n, 11, kind="box", sh_degree=0, box=(0.0, 1.0, 12.0, 18.0, 2.5, 5.5), logscale=(-4.0, 0.2))
    leaves["mean"] = leaves["mean"].copy()
    leaves["mean"][:, 0] = depth(np.random.default_rng(5)).astype(np.float32)
    leaves["opacity"] = np.full(n, 0.5, np.float32)
    return scenegen.build_tree(leaves)


def _cam(frame=0, size=(333, 211)):
    return scenegen.camera((0.0, 15.0 + 0.001 * frame, 4.0), 0.0, size[0], size[1], 0.48 * size[0])


def _run(n, equal, total):
    """`equal` leaves at one depth, the others well behind them."""
    return n, lambda r: np.concatenate([np.full(equal, 12.5), r.uniform(20.0, 24.0, total - equal)])


# (leaves, depths, replays): 256 keys are aimed at per bucket, at most 6144 fit a CTA, runs of up to 48 are ranked
CASES = {
    "one": (1, lambda r: np.full(1, 12.5), 0),
    **{"keys_%d" % n: (n, lambda r, n=n: r.uniform(10.0, 24.0, n), 0) for n in (255, 256, 257, 512, 513)},
    **{"run_%d" % k: _run(2000, k, 2000) + (0,) for k in (47, 48, 49)},
    "bucket_full": (6144, lambda r: np.full(6144, 12.5), 0),
    "bucket_too_full": (6145, lambda r: np.full(6145, 12.5), 1),
}


@pytest.mark.parametrize("name", list(CASES))
def test_bucket_edges(name):
    n, depth, replays = CASES[name]
    h = vgr.Hierarchy(_scene(n, depth))
    v, ref = vgr.View(h, pair_capacity=1 << 20), vgr.View(h, pair_capacity=1 << 20, test_hooks=RADIX_DEPTH)
    a, b = v.render(_cam(), 0.0), ref.render(_cam(), 0.0)  # tau 0: every leaf
    assert a.stats["visible_count"] == n and a.stats["replays"] == replays
    d = v.debug()
    np.testing.assert_array_equal(d["depth_order"], np.lexsort((np.arange(n), d["vis_depth"])))
    assert torch.equal(a.image(), b.image()) and a.stats["pair_count"] == b.stats["pair_count"]
    v.close(); ref.close(); h.close()


@pytest.mark.parametrize("graph", [False, True])
def test_the_partition_is_tried_again(graph):
    """64 frames by the radix passes (the replayed one among them), then one that is replayed again."""
    h = vgr.Hierarchy(_scene(9000, lambda r: np.full(9000, 12.5)))
    v, ref = vgr.View(h, pair_capacity=1 << 20, use_graph=graph), vgr.View(h, pair_capacity=1 << 20, test_hooks=RADIX_DEPTH)
    for frame in range(130):
        a, b = v.render(_cam(frame), 0.0), ref.render(_cam(frame), 0.0)
        assert a.stats["replays"] == (1 if frame % 64 == 0 else 0), frame
        assert torch.equal(a.image(), b.image())
    v.close(); ref.close(); h.close()


def test_the_partition_is_tried_again_in_a_batch():
    """Views of one batch that fall back at different frames."""
    h = vgr.Hierarchy(_scene(9000, lambda r: np.full(9000, 12.5)))
    views = [vgr.View(h, pair_capacity=1 << 20, use_graph=True) for _ in range(3)]
    ref = vgr.View(h, pair_capacity=1 << 20, test_hooks=RADIX_DEPTH)
    for k in range(3):
        for frame in range(5 * k):
            views[k].render(_cam(frame), 0.0)
    for frame in range(70):
        res = vgr.render_batch(views, [_cam(frame + k) for k in range(3)], [0.0] * 3)
        for k in range(3):
            assert res[k].stats["replays"] == (1 if (frame + 5 * k) % 64 == 0 else 0), (frame, k)
            assert torch.equal(res[k].image(), ref.render(_cam(frame + k), 0.0).image()), (frame, k)
    for x in views + [ref]:
        x.close()
    h.close()


def test_coarse_cuts_of_a_large_tree():
    """More than 2^24 nodes: a cut of a few of them is found by levels once the view
    knows that it is coarse, with a finer or unknown one by the pass; the same cuts."""
    kids = np.array([8] * sum(8 ** k for k in range(8)) + [0] * 8 ** 8, np.uint8)
    n = len(kids)
    first = np.where(kids > 0, 1 + np.cumsum(kids, dtype=np.int64) - kids, 0).astype(np.uint32)
    parent = np.concatenate([[0xFFFFFFFF], np.repeat(np.arange(n, dtype=np.uint32), kids)]).astype(np.uint32)
    mean, rad = np.zeros((n, 3), np.float32), np.zeros(n)
    lo, at, size = 0, 1, 64.0
    for level in range(9):  # an octree of cubes; radii nest with room to spare
        hi = lo + at
        if level:
            k = (np.arange(lo, hi) - lo) % 8
            off = np.stack([(k & 1) - 0.5, ((k >> 1) & 1) - 0.5, ((k >> 2) & 1) - 0.5], 1) * size
            mean[lo:hi] = mean[parent[lo:hi]] + off
        rad[lo:hi] = 2.0 * size
        lo, at, size = hi, at * 8, size / 2.0
    sc = dict(n_nodes=n, sh_degree=0, parent=parent, first_child=first, n_child=kids, mean=mean,
              cov6=np.tile(np.array([1e-2, 0, 0, 1e-2, 0, 1e-2], np.float32), (n, 1)),
              opacity=np.full(n, 0.5, np.float32), sh=np.zeros((n, 1, 3), np.float32),
              radius2=(rad ** 2).astype(np.float32), max_depth=8)
    h = vgr.Hierarchy(sc)
    v, ref = vgr.View(h), vgr.View(h, test_hooks=LOD_LEVELS)
    kernels = []
    for k, tau in enumerate((60.0, 60.0, 59.0, 12.0, 60.0)):
        cam = scenegen.camera((-80.0 + k, 0.5, 0.25), 0.0, 320, 200, 200.0)
        v.reset(), ref.reset()
        a, b = v.render(cam, tau), ref.render(cam, tau)
        assert 8 < a.cut_count < n // 32 and torch.equal(a.cut(), b.cut()) and torch.equal(a.image(), b.image())
        assert a.stats["lod_from_scratch"] == 1 and a.stats["nodes_evaluated"] == b.stats["nodes_evaluated"]
        kernels.append(a.stats["kernels"] == b.stats["kernels"])
    # the first has no last cut to go by, and tau fell to a fifth before the fourth
    assert kernels == [False, True, True, False, True]
    v.close(); ref.close(); h.close()


@pytest.mark.parametrize("offset", [1, 2, 3, 4])
@pytest.mark.parametrize("tile", [16, 32])
def test_host_images_off_a_16_byte_boundary(tiny_scene, tile, offset):
    size = (1284, 722)
    h = vgr.Hierarchy(tiny_scene)
    v = vgr.View(h, tile_size=tile)
    cam = scenegen.camera((-3.0, 10.0, 2.5), 0.0, size[0], size[1], 700.0)
    img = v.render(cam, 3.0).image().cpu().numpy().copy()
    buf = torch.full((size[0] * size[1] * 3 + 8,), -1.0, dtype=torch.float32, pin_memory=True).numpy()
    out = buf[offset:offset + img.size].reshape(img.shape)
    v.render_host(cam, 3.0, out)
    np.testing.assert_array_equal(out, img)
    assert (buf[:offset] == -1.0).all() and (buf[offset + img.size:] == -1.0).all()
    v.close(); h.close()
