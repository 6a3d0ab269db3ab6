"""Long thin diagonal Gaussians: the rounding of rho is larger than the margin of
their footprint boxes, so a pixel that looked at a record outside its box could
take it.  The blend with two pixels per lane must not: same image, evaluations
and contributions as one pixel per lane, alone and for a batch whose views blend
with one pixel per lane by themselves."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402


def _needles(n, seed=3):
    """n Gaussians of 0.3 to 6 m by 1 mm at 10 m, in planes across the view."""
    rng = np.random.default_rng(seed)
    leaves = scenegen.gen_leaves(n, seed, kind="box", sh_degree=0, box=(9.0, 11.0, -4.0, 4.0, -3.0, 3.0))
    s, a = np.exp(rng.uniform(np.log(0.3), np.log(6.0), n)), rng.uniform(0.0, np.pi, n)
    d = np.stack([0.0 * a, np.cos(a), np.sin(a)], 1)
    C = (s ** 2)[:, None, None] * d[:, :, None] * d[:, None, :] + 1e-6 * np.eye(3)
    leaves["cov6"] = np.ascontiguousarray(C[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]].astype(np.float32))
    leaves["opacity"] = np.full(n, 0.9, np.float32)
    leaves["rad2"] = scenegen.leaf_rad2(np.stack([s, s, s], 1))
    return scenegen.build_tree(leaves)


@pytest.fixture(scope="module", params=[2000, 8000])
def hier(request):
    h = vgr.Hierarchy(_needles(request.param))
    yield h
    h.close()


@pytest.mark.parametrize("tile", [16, 32])
@pytest.mark.parametrize("depth", [16, 32])
@pytest.mark.parametrize("size", [(1280, 720), (1921, 1081)])
def test_wide_equals_narrow(hier, tile, depth, size):
    narrow, wide = vgr.View(hier, tile_size=tile, blend_depth=48), vgr.View(hier, tile_size=tile, blend_depth=depth)
    for k in range(4):
        cam = scenegen.camera((0.01 * k, 0.0, 0.0), 0.002 * k, size[0], size[1], 0.57 * size[0])
        a, b = narrow.render(cam, 0.0), wide.render(cam, 0.0)
        assert torch.equal(a.image(), b.image())
        for name in ("pixel_pair_evals", "pixel_pair_contribs"):
            assert a.stats[name] == b.stats[name]
    narrow.close(); wide.close()


def test_batch_equals_alone(hier):
    size, n = (640, 360), 8
    views = [vgr.View(hier, use_graph=True) for _ in range(n)]
    cams = [scenegen.camera((0.01 * k, 0.0, 0.0), 0.002 * k, size[0], size[1], 700.0) for k in range(n)]
    res = vgr.render_batch(views, cams, [0.0] * n)
    solo = vgr.View(hier)
    for k in range(n):
        assert torch.equal(res[k].image(), solo.render(cams[k], 0.0).image()), k
    for v in views + [solo]:
        v.close()
