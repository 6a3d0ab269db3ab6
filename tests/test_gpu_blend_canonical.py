"""The canonical blend (every record at every pixel, alpha first) against an FP64
replay of the frame's own pair lists and records: image, evaluations and
contributions, at each tile size, with ragged images, lists that end inside a
chunk or a group, and pixels that stop inside one.

The bound follows the rounding of the FP32 arithmetic: with S the sum of the
magnitudes of rho's three terms, rho is off by at most 10 x 2^-24 S (offsets,
products, sums, the factor log2 e) and e^rho by another 2^-21, a relative error e
of alpha; T accumulates alpha e / (1 - alpha) + 2^-23 per record, and a colour
both.  A pixel with a decision (alpha* or stop) inside these errors is left out."""
import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

ALPHA_MIN, ALPHA_MAX, T_MIN = 1.0 / 255.0, 0.99, 1e-4


def _replay(d, W, H):
    """Per pixel: colour, its error bound, evaluations, contributions, doubt."""
    T, TW = d["tile_size"], d["tiles"][0]
    order = d["depth_order"].astype(np.int64)
    A, B, C4 = (d[k].astype(np.float64) for k in ("vis_recA", "vis_recB", "vis_rgb"))
    img, bound = np.zeros((H, W, 3)), np.zeros((H, W))
    evals, contribs = np.zeros((H, W), np.int64), np.zeros((H, W), np.int64)
    longest, doubt = np.zeros((H, W), np.int64), np.zeros((H, W), bool)
    for t, (s, e) in enumerate(d["tile_range"].astype(np.int64)):
        if e <= s:
            continue
        x0, y0 = (t % TW) * T, (t // TW) * T
        ys, xs = np.mgrid[y0:min(y0 + T, H), x0:min(x0 + T, W)]
        g = order[d["pair_rank"][s:e]]
        dx = A[g, 0] - (xs[..., None] + 0.5)
        dy = A[g, 1] - (ys[..., None] + 0.5)
        terms = [A[g, 2] * dx * dx, A[g, 3] * dx * dy, B[g, 0] * dy * dy]
        err = 10 * 2.0 ** -24 * sum(np.abs(x) for x in terms) + 2.0 ** -21
        raw = B[g, 2] * np.exp(sum(terms))
        alpha = np.minimum(ALPHA_MAX, raw)
        take = alpha >= ALPHA_MIN
        f = np.where(take, 1 - alpha, 1.0)
        after = np.cumprod(f, -1)
        rel = np.cumsum(np.where(take, alpha * err / (1 - alpha) + 2.0 ** -23, 0.0), -1)
        stop = after < T_MIN
        n = np.where(stop.any(-1), stop.argmax(-1), e - s)  # records before the stop
        idx = np.arange(e - s)
        seen = idx <= n[..., None]
        used = take & (idx < n[..., None])
        before = np.concatenate([np.ones_like(after[..., :1]), after[..., :-1]], -1)
        w = np.where(used, alpha * before, 0.0)
        sl = np.s_[y0:y0 + ys.shape[0], x0:x0 + xs.shape[1]]
        img[sl] = np.einsum("yxn,nc->yxc", w, C4[g, :3])
        bound[sl] = (w * np.abs(C4[g, :3]).max(-1) * (err + rel + (idx + 2) * 2.0 ** -24)).sum(-1)
        evals[sl], contribs[sl], longest[sl] = np.minimum(n + 1, e - s), used.sum(-1), e - s
        doubt[sl] = (seen & ((np.abs(raw / ALPHA_MIN - 1) <= err) |
                             (take & (np.abs(after / T_MIN - 1) <= rel)))).any(-1)
    return img, bound, evals, contribs, longest, doubt


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("n,scale,opacity", [(1, 1.0, 1.0), (37, 0.5, 8.0), (600, -1.0, 1.0), (600, 0.5, 8.0)])
def test_canonical_blend_follows_the_lists(tile, n, scale, opacity):
    W, H = 203, 117
    leaves = scenegen.gen_leaves(n, 5, kind="box", sh_degree=0, box=(4.0, 12.0, 10.0, 20.0, 0.0, 8.0),
                                 logscale=(scale, 0.5), opacity_sigma=opacity)
    h = vgr.Hierarchy(scenegen.build_tree(leaves))
    v = vgr.View(h, filter=vgr.FILTER_CANONICAL, tile_size=tile)
    r = v.render(scenegen.camera((-3.0, 15.0, 4.0), 0.0, W, H, 0.6 * W), 0.0)
    got = r.image().cpu().numpy().astype(np.float64)
    img, bound, evals, contribs, longest, doubt = _replay(v.debug(), W, H)
    assert doubt.mean() < 0.05
    assert (np.abs(got - img).max(-1) <= bound + 1e-9)[~doubt].all()
    slack = int(longest[doubt].sum())
    assert abs(r.stats["pixel_pair_evals"] - int(evals.sum())) <= slack
    assert abs(r.stats["pixel_pair_contribs"] - int(contribs.sum())) <= slack
    v.close(); h.close()
