"""The emission of items of 512 tiles and more, which several warps share by ranges of row bands: every listed
(tile, item) pair once and in depth order, whole and cut lists, kept and rebuilt, one view and several, and the
images those of tiles four times as large, at which next to no item has that many."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


def _scene(n, opacity, seed):
    sc = S.random_scene(n, 1024, 512, seed=seed, sh_degree=0, radius=(1.0, 3.0), log_scale=(-0.6, 0.9))
    sc.opacity[:] = opacity
    sc.means[: n // 8, ::2] *= 0.01  # near the poles: footprints of whole tile rows
    sc.scales[n // 2:] *= 0.02       # and small ones among them
    return sc


@pytest.mark.parametrize("full", [0, 1])
@pytest.mark.parametrize("opacity", [0.02, 0.9])
@pytest.mark.parametrize("views", [1, 2])
def test_pairs_and_images(views, opacity, full):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = _scene(4000, opacity, 31)
    p = to_torch(sc)
    vs = [S.yaw_view(1024, 512, (0.05 * k, 0.0, 0.1), 0.8 * k) for k in range(views)]
    gen = torch.Generator("cuda").manual_seed(3)
    w = [torch.randn(3, 512, 1024, device="cuda", generator=gen) for _ in vs]
    out = []
    for kw in (dict(), dict(recompute_lists=True), dict(tile_w=32, tile_h=32)):
        r = Rasterizer()
        imgs, _ = r.forward(*p, vs, RenderSettings(sh_degree=0, full_lists=full, **kw))
        st = r.stats()
        assert st["status"] == 0
        d = r.debug_lists()
        place = np.empty(len(d["depth_items"]), np.int64)
        place[d["depth_items"]] = np.arange(len(place))
        words = d["pair_tiles"].astype(np.int64) * len(place) + place[d["pair_items"]]
        assert len(words) == st["pairs_sorted"] and np.all(words[1:] > words[:-1])
        if full:
            assert st["pairs_sorted"] == st["pairs"]
        if not kw:
            count = np.bincount(d["pair_items"], minlength=len(place))
            assert (count >= 512).sum() > (0 if opacity > 0.5 and not full else 100)
        r.backward(w)  # rebuilds the lists where they were not kept
        again = r.debug_lists()
        assert r.status() == 0 and all(np.array_equal(d[k], again[k]) for k in d)
        out.append(imgs)
    for imgs in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], imgs))
