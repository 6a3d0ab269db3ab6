"""The blend with two pixels per lane (launches with many strips) against the
one with one (48 hits staged per chunk keep it): the same image bit for bit and
the same statistics, on images whose last columns, rows and strips are ragged,
at both tile sizes, with host images, the full strip walk and a batch."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

SIZES = [(1280, 720), (1283, 721), (1301, 1003), (2049, 1089), (1922, 1070)]
FULL_WALK = 2  # VGR_HOOK_FULL_STRIP_WALK


@pytest.fixture(scope="module")
def hier(small_sh3_scene):
    h = vgr.Hierarchy(small_sh3_scene)
    yield h
    h.close()


def _cam(k, size):
    return scenegen.camera((2.0 + 0.1 * k, 15.0, 3.0), 0.2 + 0.02 * k, size[0], size[1], 0.8 * size[0])


@pytest.mark.parametrize("tile", [16, 32])
@pytest.mark.parametrize("size", SIZES)
def test_wide_equals_narrow(hier, tile, size):
    narrow = vgr.View(hier, tile_size=tile, blend_depth=48)
    views = [vgr.View(hier, tile_size=tile, blend_depth=d, use_graph=g, test_hooks=k)
             for d, g, k in ((32, False, 0), (16, True, 0), (32, True, FULL_WALK))]
    for k in range(2):
        ref = narrow.render(_cam(k, size), 2.0)
        img = ref.image().clone()
        assert float(img.max()) > 0.1
        for v in views:
            r = v.render(_cam(k, size), 2.0)
            assert torch.equal(r.image(), img)
            assert r.stats["pixel_pair_contribs"] == ref.stats["pixel_pair_contribs"]
            if v is not views[2]:
                assert r.stats["pixel_pair_evals"] == ref.stats["pixel_pair_evals"]
        out = torch.zeros((size[1], size[0], 3), dtype=torch.float32, pin_memory=True).numpy()
        views[0].render_host(_cam(k, size), 2.0, out)
        np.testing.assert_array_equal(out, img.cpu().numpy())
    for v in views + [narrow]:
        v.close()


def test_opaque_pixels_stop_alike(hier):
    """A camera close to many large, nearly opaque Gaussians: most pixels stop early."""
    leaves = scenegen.gen_leaves(4000, 21, kind="box", sh_degree=1, box=(0.0, 10.0, 0.0, 10.0, 0.0, 10.0),
                                 logscale=(-0.5, 0.3), opacity_sigma=8.0)
    h = vgr.Hierarchy(scenegen.build_tree(leaves))
    cam = scenegen.camera((-6.0, 5.0, 5.0), 0.0, 1363, 769, 900.0)
    va, vb = vgr.View(h, blend_depth=48), vgr.View(h)
    a, b = va.render(cam, 0.0), vb.render(cam, 0.0)
    assert torch.equal(a.image(), b.image())
    for k in ("pixel_pair_evals", "pixel_pair_contribs"):
        assert a.stats[k] == b.stats[k]
    va.close(); vb.close(); h.close()


def test_batch_of_small_views_blends_wide(hier):
    """Views too small for it alone reach it together, with the same images."""
    n, size = 8, (640, 360)
    views = [vgr.View(hier, use_graph=True) for _ in range(n)]
    solo = vgr.View(hier)
    res = vgr.render_batch(views, [_cam(i, size) for i in range(n)], [2.0] * n)
    for i in range(n):
        r = solo.render(_cam(i, size), 2.0)
        assert torch.equal(res[i].image(), r.image()), i
        assert res[i].stats["pixel_pair_evals"] == r.stats["pixel_pair_evals"]
    for v in views + [solo]:
        v.close()
