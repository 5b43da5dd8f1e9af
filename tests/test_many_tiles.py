"""Frames on either side of 65536 tiles, from which on the tile sort takes a third pass and clears its own scratch:
repeated and replayed binnings and rebuilt lists give the image and the gradients of larger tiles."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("height", [1024, 1028, 2048])  # 65536, 65792 and 131072 tiles of 8 x 4
def test_repeated_binnings_and_rebuilt_lists(height, full):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(4000, 2048, height, seed=51, sh_degree=0, radius=(1.0, 4.0), log_scale=(-4.0, 0.8))
    p, w = to_torch(sc), [torch.randn(3, height, 2048, device="cuda", generator=torch.Generator("cuda").manual_seed(1))]
    ref = Rasterizer()
    (want,), _ = ref.forward(*p, sc.views, RenderSettings(sh_degree=0, tile_w=32, tile_h=16))
    grads = ref.backward(w)
    rs = RenderSettings(sh_degree=0, tile_w=8, tile_h=4, full_lists=full, recompute_lists=True)
    r = Rasterizer()
    (img,), _ = r.forward(*p, sc.views, rs)
    assert torch.equal(img, want)
    r.capacity_mode = "fixed"
    r.bin_sort()
    (img,), _ = r.render_fwd(want_T=False)
    assert torch.equal(img, want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.preprocess(*p, sc.views, rs)
        r.bin_sort()
        (img,), _ = r.render_fwd(want_T=False)
    for _ in range(2):
        img.zero_()
        g.replay()
        assert torch.equal(img, want)
        got = r.backward(w)
        assert r.status() == 0
        for name in GRAD_NAMES:  # the same terms: only the order of the additions differs
            a, b = (x[name].cpu().numpy().astype(np.float64) for x in (got, grads))
            assert rel_l2(a, b) < 1e-5, name
