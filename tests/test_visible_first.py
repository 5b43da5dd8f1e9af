"""Perspective frames of many items partition them before the depth sort: the depth order is the whole
sort's (visible items by key and item, then the culled ones in item order), for counts around the partition's
tiles, repeated and replayed binnings and rebuilt lists, and the images are the single views'."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


def _frame(n, seed):
    sc = S.random_scene(n, 96, 96, seed=seed, sh_degree=0, radius=(0.1, 5.0), log_scale=(-4.5, 0.5))
    return sc, S.cubemap_views(96, (0.1, 0.0, -0.2))


def _check_order(d):
    k, i = d["depth_keys"], d["depth_items"]
    assert np.array_equal(np.sort(i), np.arange(len(i)))
    assert np.all((k[1:] > k[:-1]) | ((k[1:] == k[:-1]) & (i[1:] > i[:-1])))
    return int((k != 0xFFFFFFFF).sum())


@pytest.mark.parametrize("n", [21846, 22187, 30000, 100_001])  # 131076 items and up; 65 * 2048 + 2
def test_order_and_images(n):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc, views = _frame(n, n)
    rs, p = RenderSettings(sh_degree=0), to_torch(sc)
    r = Rasterizer()
    imgs, _ = r.forward(*p, views, rs)
    st = r.stats()
    assert st["status"] == 0
    assert _check_order(r.debug_lists()) == st["visible"] < 0.5 * 6 * n
    for k, v in enumerate(views):  # one view: too few items for the partition
        (one,), _ = Rasterizer().forward(*p, [v], rs)
        assert torch.equal(imgs[k], one), k
    again, _ = r.forward(*p, views, rs)
    r.bin_sort()  # repeated
    twice, _ = r.render_fwd(want_T=False)
    assert all(torch.equal(a, b) and torch.equal(a, c) for a, b, c in zip(imgs, again, twice))
    _check_order(r.debug_lists())
    r.capacity_mode = "fixed"
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):  # the binning alone, replayed
        r.bin_sort()
    for _ in range(2):
        g.replay()
        out, _ = r.render_fwd(want_T=False)
        torch.cuda.synchronize()
        assert r.status() == 0 and all(torch.equal(a, b) for a, b in zip(imgs, out))


def test_all_culled_mixed_views_and_rebuilt_lists():
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc, faces = _frame(50_000, 9)
    p = to_torch(sc)
    far = [t.clone() for t in p]
    far[3].fill_(0.001)  # below 1 / 255 everywhere
    r = Rasterizer()
    imgs, _ = r.forward(*far, faces, RenderSettings(sh_degree=0, bg=(0.25, 0.5, 0.75)))
    assert r.stats()["visible"] == 0 and all(float(i[1].min()) == float(i[1].max()) == 0.5 for i in imgs)
    views = [faces[0], S.yaw_view(96, 48, (0.1, 0.0, -0.2), 0.3), faces[3]]
    w = [torch.randn(3, v.height, v.width, device="cuda", generator=torch.Generator("cuda").manual_seed(k))
         for k, v in enumerate(views)]
    out = []
    for rebuild in (False, True):
        r = Rasterizer()
        imgs, _ = r.forward(*p, views, RenderSettings(sh_degree=0, recompute_lists=rebuild))
        _check_order(r.debug_lists())
        out.append((imgs, r.backward(w)))
    for k, v in enumerate(views):
        (one,), _ = Rasterizer().forward(*p, [v], RenderSettings(sh_degree=0))
        assert torch.equal(out[0][0][k], one) and torch.equal(out[1][0][k], one)
    for name in GRAD_NAMES:
        a, b = (o[1][name].cpu().numpy().astype(np.float64) for o in out)
        assert rel_l2(a, b) < 1e-6, name
