"""The temporal update over frames whose granularity test is not monotone: the
update cannot see every such frame, and leaves a node and its descendant in one
cut, so the next update reports nodes twice.  The lists of that frame must still
be the cut: ascending, every node once, equal to the top-down traversal's, with
thousands of nodes behind the ones reported twice."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

LOD_LEVELS = 8  # VGR_HOOK_LOD_LEVELS


def _scene():
    """Root 0; under it A = 1 and D = 2.  A's children are B = 3, whose child is a
    leaf, and the leaf C = 4; D's subtree has 32,768 leaves five levels down.  Seen
    from x = 0 B expands and A, whose radius falls short of nesting by less than the
    tolerance of the loader, does not."""
    rng = np.random.default_rng(4)
    parent, first, kids, mean, rad = [0xFFFFFFFF], [0], [2], [(20.0, 0.0, 0.0)], [1000.0]

    def add(p, m, r):
        if first[p] == 0:
            first[p] = len(parent)
        parent.append(p); first.append(0); kids.append(0); mean.append(m); rad.append(r)
        return len(parent) - 1

    a = add(0, (19.99999, 0, 0), 19.999985)
    d = add(0, (40.0, 0, 0), 200.0)
    kids[a], kids[d] = 2, 8
    b = add(a, (9.99999, 0, 0), 10.0)
    add(a, (12.0, 0.5, 0.2), 0.5)
    kids[b] = 1
    level = [add(d, (40.0, 0, 0), 200.0) for _ in range(8)]
    add(b, (9.99999, 0.3, 0.1), 1.0)
    for depth in range(4):
        nxt = []
        for p in level:
            kids[p] = 8
            for _ in range(8):
                leaf = depth == 3
                m = (rng.uniform(8, 60), rng.uniform(-3, 3), rng.uniform(-2, 2)) if leaf else (40.0, 0, 0)
                nxt.append(add(p, m, 0.1 if leaf else 200.0))
        level = nxt
    n = len(parent)
    mean, r2 = np.array(mean, np.float32), (np.array(rad, np.float64) ** 2).astype(np.float32)
    sc = dict(n_nodes=n, sh_degree=0, parent=np.array(parent, np.uint32), first_child=np.array(first, np.uint32),
              n_child=np.array(kids, np.uint8), mean=mean,
              cov6=np.tile(np.array([1e-3, 0, 0, 1e-3, 0, 1e-3], np.float32), (n, 1)),
              opacity=np.full(n, 0.5, np.float32), sh=rng.normal(size=(n, 1, 3)).astype(np.float32), radius2=r2,
              max_depth=6)
    sc["bbox"] = scenegen.tree_boxes(sc)
    assert mean[b, 0] ** 2 < r2[b] and mean[a, 0] ** 2 >= r2[a]  # the child expands, its parent does not
    return sc


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("kw", [dict(), dict(lod_frustum=True), dict(lod_interp=True)])
def test_lists_after_a_missed_frame(kw, graph):
    h = vgr.Hierarchy(_scene())
    v, ref = vgr.View(h, use_graph=graph, **kw), vgr.View(h, test_hooks=LOD_LEVELS, temporal=False, **kw)
    # A open, then the frame the update misses, A open again (its leaf is reported by
    # A's subtree and as a staying node), and A and B shut behind another missed
    # frame (A is reported by the collapsing leaf and as a staying node)
    for x in (0.001, 0.0, 0.001, 0.001, 0.0, -0.001, 0.001, 0.0, 0.001):
        cam = scenegen.camera((x, 0.0, 0.0), 0.0, 640, 360, 640.0)
        r, s = v.render(cam, 640.0), ref.render(cam, 640.0)  # tau = f: a node expands when the camera is in its sphere
        cut = r.cut().cpu().numpy().view(np.uint32)
        assert len(cut) == r.cut_count and (np.diff(cut.astype(np.int64)) > 0).all()
        if x == 0.0:
            continue  # A's leaf may stay in the cut with A
        np.testing.assert_array_equal(cut, s.cut().cpu().numpy().view(np.uint32))
        assert r.stats["front_count"] == s.stats["front_count"] and r.stats["visible_count"] > 20000
        np.testing.assert_array_equal(v.debug()["vis_node"], ref.debug()["vis_node"])
        assert torch.equal(r.image(), s.image())
    v.close(); ref.close(); h.close()


def test_nodes_that_no_traversal_reaches_overflow_nothing():
    """A tree whose cut is one node, with 2^24 leaves behind a child that expands while
    its parent does not: the pass over the nodes lists them all, more than a frame may
    have in front of the camera, and the traversal that follows finds the cut."""
    kids = [1, 1] + [8] * sum(8 ** k for k in range(8)) + [0] * 8 ** 8  # root, A, then an octree under B
    n = len(kids)
    kids = np.array(kids, np.uint8)
    first = np.where(kids > 0, 1 + np.cumsum(kids, dtype=np.int64) - kids, 0).astype(np.uint32)
    parent = np.concatenate([[0xFFFFFFFF], np.repeat(np.arange(n, dtype=np.uint32), kids)]).astype(np.uint32)
    x = np.full(n, 9.99999, np.float32)
    x[:2] = 19.99999
    r2 = np.where(kids > 0, np.float32(100.0), np.float32(1e-4)).astype(np.float32)
    r2[0], r2[1] = 100.0 ** 2, np.float32(19.999985 ** 2)
    sc = dict(n_nodes=n, sh_degree=0, parent=parent, first_child=first, n_child=kids,
              mean=np.stack([x, 0 * x, 0 * x], 1), cov6=np.tile(np.array([1e-3, 0, 0, 1e-3, 0, 1e-3], np.float32), (n, 1)),
              opacity=np.full(n, 0.8, np.float32), sh=np.zeros((n, 1, 3), np.float32), radius2=r2, max_depth=10)
    h = vgr.Hierarchy(sc)
    v = vgr.View(h)
    r = v.render(scenegen.camera((0.0, 0.0, 0.0), 0.0, 64, 48, 64.0), 64.0)
    assert r.cut().cpu().tolist() == [1] and r.stats["front_count"] == 1
    assert r.stats["replays"] == 1 and r.stats["lod_from_scratch"] == 1
    v.close(); h.close()
