"""Scenes with a few leaves far outside the others, as trained scenes have them:
the depth partition must keep its bins for the frame's depths.  The same kernels
run, with as few replays, as without those leaves, and the order is the
definition's, near and far ones included."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402


def _scene(n, far, distance):
    """n leaves 14 to 30 m in front of the camera, `far` of them `distance` away in all directions."""
    leaves = scenegen.gen_leaves(n, 2, kind="box", sh_degree=0, box=(0.0, 16.0, 0.0, 16.0, 0.0, 4.0), logscale=(-5.0, 0.5))
    if far:
        d = np.random.default_rng(9).normal(size=(far, 3))
        leaves["mean"] = leaves["mean"].copy()
        leaves["mean"][:far] = distance * d / np.linalg.norm(d, axis=1, keepdims=True)
    return scenegen.build_tree(leaves)


@pytest.mark.parametrize("far,distance", [(10, 1e6), (10, 1e4), (20000, 1e5)])
def test_outliers_cost_no_bins(far, distance):
    n, seen = 2_000_000, {}
    for k in (0, far):
        h = vgr.Hierarchy(_scene(n, k, distance))
        v = vgr.View(h)
        r = [v.render(scenegen.camera((-14.0 + 0.01 * f, 8.0, 2.0), 0.0, 960, 540, 550.0), 0.0) for f in range(2)][1]
        assert r.stats["visible_count"] > 0.95 * n and r.stats["replays"] == 0  # (the first frame grows buffers)
        seen[k] = r.stats["kernels"]
        d = v.debug()
        want = np.lexsort((np.arange(d["n_visible"]), d["vis_depth"]))
        np.testing.assert_array_equal(d["depth_order"], want)
        v.close(); h.close()
    assert seen[far] == seen[0]  # no radix passes
