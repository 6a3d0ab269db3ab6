"""The depth order by partition and per-bucket sort (k_depth.cu) against the
definition -- (FP32 depth key, in-front index) ascending -- and against the
radix passes, at the sizes where it can go wrong: a handful of Gaussians, the
edges of a bucket, many equal depths (the bitonic buckets), depths too
concentrated for any bucket (replay with the radix passes), duplicates at every
depth, a second frame on the same buffers."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

RADIX_DEPTH = 4  # VGR_HOOK_RADIX_DEPTH


def _scene(n, depth):
    """n leaves in a 30 x 30 x 8 m box whose x is depth(rng, n): the camera looks along +x."""
    leaves = scenegen.gen_leaves(n, 11, kind="box", sh_degree=1, box=(0.0, 30.0, 0.0, 30.0, 0.0, 8.0),
                                 logscale=(-3.5, 0.3))
    rng = np.random.default_rng(5)
    leaves["mean"] = leaves["mean"].copy()
    leaves["mean"][:, 0] = depth(rng, n).astype(np.float32)
    return scenegen.build_tree(leaves)


CASES = {
    "one": (1, lambda r, n: np.full(n, 10.0), 0),
    "few": (7, lambda r, n: r.uniform(1.0, 20.0, n), 0),
    "bucket_edge": (257, lambda r, n: r.uniform(1.0, 20.0, n), 0),
    "rows": (4097, lambda r, n: np.exp(r.uniform(0.0, 4.0, n)), 0),
    "many": (120000, lambda r, n: r.uniform(0.5, 30.0, n), 0),
    "equal_fits": (6000, lambda r, n: np.full(n, 12.5), 0),
    "equal_skew": (30000, lambda r, n: np.full(n, 12.5), 1),
    "eight_depths": (40000, lambda r, n: r.integers(2, 10, n) * 2.5, 0),
    "far_outlier": (20000, lambda r, n: np.where(np.arange(n) == 0, 3.0e6, r.uniform(9.0, 9.5, n)), None),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("half", [False, True])
def test_order(name, half):
    n, depth, replays = CASES[name]
    h = vgr.Hierarchy(_scene(n, depth), vgr.STORE_HALF if half else vgr.STORE_FP32)
    v, ref = vgr.View(h, use_graph=True), vgr.View(h, test_hooks=RADIX_DEPTH)
    for frame in range(3):
        cam = scenegen.camera((0.0, 15.0 + 0.01 * frame, 4.0), 0.0, 333, 211, 160.0)
        a, b = v.render(cam, 0.0), ref.render(cam, 0.0)  # tau 0: every leaf
        if replays is not None:
            assert a.stats["replays"] == (replays if frame == 0 else 0)
        for k in ("visible_count", "pair_count", "candidate_pairs", "pixel_pair_contribs"):
            assert a.stats[k] == b.stats[k], k
        assert a.stats["visible_count"] > 0 or n == 1  # the single leaf lies outside the image
        assert torch.equal(a.image(), b.image())
        da, db = v.debug(), ref.debug()
        want = np.lexsort((np.arange(da["n_visible"]), da["vis_depth"]))  # vis_* are in ascending node id
        np.testing.assert_array_equal(da["depth_order"], want)
        np.testing.assert_array_equal(db["depth_order"], want)
    v.close(); ref.close(); h.close()


@pytest.mark.parametrize("n,equal", [(300_000, 0), (700_000, 3500), (1_400_000, 0), (1_400_000, 4000)])
def test_order_of_large_frames(n, equal):
    """More keys than one small bucket per CTA: buckets sized by whole rounds of
    CTAs, and by the room that a bin of many equal depths leaves."""
    def depth(r, m):
        x = r.uniform(20.0, 60.0, m)
        x[:equal] = 40.0
        return x
    h = vgr.Hierarchy(_scene(n, depth))
    v = vgr.View(h)
    r = v.render(scenegen.camera((0.0, 15.0, 4.0), 0.0, 333, 211, 160.0), 0.0)
    d = v.debug()
    assert r.stats["replays"] <= 1 and r.stats["visible_count"] > 0.9 * n  # (one for the pair buffer, if any)
    want = np.lexsort((np.arange(d["n_visible"]), d["vis_depth"]))
    np.testing.assert_array_equal(d["depth_order"], want)
    v.close(); h.close()
