"""Key counts at the edges of the pair sort's tiles: a tile holds 1024 keys up to
152 x 1024 keys and 4096 above, so the edges lie where a tile, a group of 32
tiles, or the tile size changes.  Keys at random, in runs of one digit and of few
digits.  Stable, against numpy's stable sort: whole
numbers, equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_02774_gb300 as vgr  # noqa: E402

SMALL = 152 * 1024


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 32 * 1024, 32 * 1024 + 1, SMALL - 1, SMALL, SMALL + 1,
                               39 * 4096, 64 * 4096 + 1, 304 * 4096, 304 * 4096 + 5])
@pytest.mark.parametrize("key_bits,kind", [(8, "random"), (19, "random"), (19, "runs"), (19, "few")])
def test_sort_at_tile_size_edges(n, key_bits, kind):
    rng = np.random.default_rng(n + key_bits)
    keys = rng.integers(0, 1 << key_bits, n, dtype=np.uint32)
    if kind == "runs":  # of one digit, across warps and tiles
        keys = (np.arange(n, dtype=np.uint32) // 45) & 0x7FFFF
    elif kind == "few":  # few digits in every pass
        keys = keys % 5 * 0x10101
    vals = np.arange(n, dtype=np.uint32)
    order = np.argsort(keys, kind="stable")
    k = torch.from_numpy(keys.view(np.int32)).cuda()
    v = torch.from_numpy(vals.view(np.int32)).cuda()
    ko, vo = vgr.sort_pairs(k, v, key_bits)
    torch.cuda.synchronize()
    assert np.array_equal(ko.cpu().numpy().view(np.uint32), keys[order])
    assert np.array_equal(vo.cpu().numpy().view(np.uint32), vals[order])
