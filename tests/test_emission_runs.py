"""The pair emission at the edges of its run lists: tile rows of 2048 tiles (the most there are) with
footprints across the seam and around the poles, items of 32 and 33 tiles and of 6 and 7 bands, and pairs
beyond the capacity. The image does not depend on the tile shape, so every shape has to give the same one."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


def _image(sc, **kw):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    r = Rasterizer()
    (img,), _ = r.forward(*to_torch(sc), sc.views, RenderSettings(sh_degree=0, **kw), want_T=False)
    torch.cuda.synchronize()
    assert r.status() == 0
    return img.cpu().numpy(), r


@pytest.mark.parametrize("full", [False, True])
def test_widest_rows(full):
    sc = S.random_scene(400, 16384, 40, seed=31, sh_degree=0, log_scale=(-3.0, 1.0))
    sc.means[:40, 0] *= 0.02  # behind the camera on the seam, some across both poles
    sc.means[:40, 2] = -np.abs(sc.means[:40, 2])
    sc.means[40:80, [0, 2]] *= 0.05
    ref, _ = _image(sc, tile_w=32, tile_h=16, full_lists=True)
    for tw, th in ((8, 8), (8, 4), (16, 6)):
        assert np.array_equal(_image(sc, tile_w=tw, tile_h=th, full_lists=full)[0], ref), (tw, th)


def test_item_sizes_around_the_limits():
    sc = S.random_scene(3000, 512, 256, seed=32, sh_degree=0, log_scale=(-2.2, 0.9))
    ref, r = _image(sc, tile_w=32, tile_h=32, full_lists=True)
    img, r = _image(sc, tile_w=8, tile_h=8, full_lists=True)
    assert np.array_equal(img, ref)
    items = r.debug_lists()["pair_items"]
    sizes = np.bincount(items)
    assert all((sizes == k).any() for k in (1, 31, 32, 33, 34)) and sizes.max() > 300
    # every shape and the cut lists
    for tw, th in ((16, 16), (32, 8), (8, 16)):
        assert np.array_equal(_image(sc, tile_w=tw, tile_h=th)[0], ref), (tw, th)


@pytest.mark.parametrize("drop", [1, 33, 1000])
def test_capacity_keeps_a_prefix(drop):
    """Pairs beyond the capacity are dropped from the end of the depth order."""
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(3000, 512, 256, seed=32, sh_degree=0, log_scale=(-2.2, 0.9))
    rs = RenderSettings(sh_degree=0, tile_w=8, tile_h=8, full_lists=True)
    whole = Rasterizer()
    whole.forward(*to_torch(sc), sc.views, rs)
    pairs, full = whole.stats()["pairs"], whole.debug_lists()
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(pairs - drop)
    r.forward(*to_torch(sc), sc.views, rs)
    torch.cuda.synchronize()
    assert r.status() == 1 and r.stats()["pairs_sorted"] == pairs - drop
    cut = r.debug_lists()
    rank = np.empty(len(full["depth_items"]), np.int64)
    rank[full["depth_items"]] = np.arange(len(rank))

    def in_emission_order(d):  # by the item's place in the depth order, then row-major tiles per item
        return sorted(zip(rank[d["pair_items"]], d["pair_tiles"]))

    last = rank[cut["pair_items"]].max()
    a, b = in_emission_order(full), in_emission_order(cut)
    assert [p for p in a if p[0] < last] == [p for p in b if p[0] < last]
    assert set(b) <= set(a)
