"""The binning's scratch and list choices: a frame of few pairs keeps its whole lists once its pairs have
been read back (same image as the cut lists), the sorts' scratch is clear for a repeated odgs_bin_sort
and for replays of a captured one, and the block scan covers frames of more than one step."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


def _image(r):
    import torch
    imgs, _ = r.render_fwd(want_T=False)
    torch.cuda.synchronize()
    return [i.cpu().numpy() for i in imgs]


def test_few_pairs_keep_whole_lists():
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(3000, 256, 128, seed=21, sh_degree=1, radius=(1.0, 4.0), log_scale=(-2.5, 0.8))
    rs, p = RenderSettings(sh_degree=1), to_torch(sc)
    r = Rasterizer()
    r.preprocess(*p, sc.views, rs)
    r.bin_sort()
    whole, st = _image(r), r.stats()
    assert st["pairs_sorted"] == st["pairs"] <= 32768
    f = Rasterizer(capacity_mode="fixed")  # pairs unknown to the host: cut lists
    f.reserve_pairs(st["pairs"])
    f.preprocess(*p, sc.views, rs)
    f.bin_sort()
    assert np.array_equal(_image(f)[0], whole[0]) and f.stats()["pairs_sorted"] <= st["pairs"]
    # known, but not all would fit: the cut lists, as before
    cut = f.stats()["pairs_sorted"]
    small = Rasterizer(capacity_mode="fixed")
    small.reserve_pairs(st["pairs"] - 1)
    small.preprocess(*p, sc.views, rs)
    assert small.query_pairs() == st["pairs"]
    small.bin_sort()
    assert small.stats()["pairs_sorted"] == min(cut, st["pairs"] - 1)
    if cut < st["pairs"]:
        assert np.array_equal(_image(small)[0], whole[0]) and small.status() == 0


@pytest.mark.parametrize("n,full", [(900, False), (9000, False), (9000, True)])
def test_repeated_and_replayed_binning(n, full):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(n, 256, 128, seed=22, sh_degree=0, log_scale=(-2.4, 0.6))
    rs, p = RenderSettings(sh_degree=0, full_lists=full), to_torch(sc)
    r = Rasterizer()
    r.preprocess(*p, sc.views, rs)
    r.bin_sort()
    ref = _image(r)[0]
    r.bin_sort()  # the depth order of the first is sorted again
    assert np.array_equal(_image(r)[0], ref)
    r.capacity_mode = "fixed"
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        r.preprocess(*p, sc.views, rs)
        r.bin_sort()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):  # the binning alone
        r.bin_sort()
    for _ in range(3):
        g.replay()
        torch.cuda.synchronize()
        assert r.status() == 0
        assert np.array_equal(_image(r)[0], ref)


def test_scan_of_many_blocks():
    """16 views of 300K Gaussians: 9375 blocks of 512 items, more than one step of the scan (8192)."""
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(300_000, 64, 32, seed=23, sh_degree=0, log_scale=(-5.0, 0.5))
    views = [S.yaw_view(64, 32, (0.1 * i, 0.0, 0.0), 0.4 * i) for i in range(16)]
    rs, p = RenderSettings(sh_degree=0), to_torch(sc)
    r = Rasterizer()
    r.preprocess(*p, views, rs)
    r.bin_sort()
    imgs = _image(r)
    for k in (0, 7, 15):
        one = Rasterizer()
        one.preprocess(*p, [views[k]], rs)
        one.bin_sort()
        assert np.array_equal(_image(one)[0], imgs[k]), k
