"""The from-scratch cut by one pass over all the nodes (k_lod_dense) against the
level-by-level traversal and the oracle: same cut, same images, same number of
nodes evaluated, at tree sizes around its rows, for the frustum-aware and the
interpolated variants; and a tree whose granularity test is not monotone, which
the pass has to leave to the traversal."""
import numpy as np
import pytest

import oracle
import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

LOD_LEVELS = 8  # VGR_HOOK_LOD_LEVELS


@pytest.mark.parametrize("n", [1, 5, 700, 5000, 60000])
@pytest.mark.parametrize("kw", [dict(), dict(lod_frustum=True), dict(lod_interp=True),
                                dict(lod_frustum=True, lod_interp=True), dict(filter=vgr.FILTER_CANONICAL)])
def test_dense_equals_levels(n, kw):
    leaves = scenegen.gen_leaves(n, 31, kind="box", sh_degree=1, box=(0.0, 40.0, 0.0, 40.0, 0.0, 8.0),
                                 logscale=(-2.5, 0.4))
    sc = scenegen.build_tree(leaves)
    h = vgr.Hierarchy(sc)
    v, ref = vgr.View(h, use_graph=True, **kw), vgr.View(h, test_hooks=LOD_LEVELS, **kw)
    cams = [scenegen.camera((2.0, 20.0, 3.0), 0.1, 320, 200, 200.0), scenegen.camera((35.0, 5.0, 4.0), 2.0, 320, 200, 200.0),
            scenegen.camera((-80.0, 20.0, 4.0), 0.0, 320, 200, 200.0)]
    for tau in (0.0, 2.0, 9.0):
        for cam in cams:
            v.reset(), ref.reset()
            a, b = v.render(cam, tau), ref.render(cam, tau)
            assert a.stats["lod_from_scratch"] == b.stats["lod_from_scratch"] == 1
            assert a.stats["replays"] == b.stats["replays"]  # (a pair buffer that grows)
            for k in ("cut_count", "front_count", "visible_count", "nodes_evaluated", "pair_count"):
                assert a.stats[k] == b.stats[k], (k, tau)
            assert torch.equal(a.cut(), b.cut())
            assert torch.equal(a.image(), b.image())
            if not kw:
                np.testing.assert_array_equal(a.cut().cpu().numpy().view(np.uint32), oracle.render(sc, cam, tau)["cut"])
            # the temporal update that follows starts from the same cut
            a, b = v.render(cams[0], tau), ref.render(cams[0], tau)
            assert torch.equal(a.cut(), b.cut())
    v.close(); ref.close(); h.close()


def test_test_not_monotone():
    """Root, node, inner child, leaf on a line: seen from x = 0 the inner child
    expands and its parent, whose radius falls short of nesting by less than the
    tolerance of the loader, does not.  The cut stops at the parent."""
    x = np.array([19.99999, 19.99999, 9.99999, 9.99999], np.float32)
    r2 = np.array([100.0 ** 2, 19.999985 ** 2, 100.0, 1.0], np.float32)
    sc = dict(n_nodes=4, sh_degree=0, parent=np.array([0xFFFFFFFF, 0, 1, 2], np.uint32),
              first_child=np.array([1, 2, 3, 0], np.uint32), n_child=np.array([1, 1, 1, 0], np.uint8),
              mean=np.stack([x, 0 * x, 0 * x], 1), cov6=np.tile(np.array([0.1, 0, 0, 0.1, 0, 0.1], np.float32), (4, 1)),
              opacity=np.full(4, 0.8, np.float32), sh=np.zeros((4, 1, 3), np.float32), radius2=r2, max_depth=3)
    assert x[2] ** 2 < r2[2] and x[1] ** 2 >= r2[1]  # the child expands, its parent does not
    h = vgr.Hierarchy(sc)
    v = vgr.View(h, use_graph=True)
    cam = scenegen.camera((0.0, 0.0, 0.0), 0.0, 64, 48, 64.0)
    for frame in range(3):
        v.reset()
        r = v.render(cam, 64.0)  # tau = f: a node expands when the camera is inside its sphere
        assert r.cut().cpu().tolist() == [1]
        assert r.stats["replays"] == (1 if frame == 0 else 0) and r.stats["lod_from_scratch"] == 1
        assert r.stats["nodes_evaluated"] == 2
    v.close(); h.close()
