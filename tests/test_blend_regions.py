"""Blend kernels' per-warp entry walks: every tile shape, region shape and number of pixels per thread
gives the same image bit for bit and the same gradients, on a view that stress the footprint test
(clusters at the seam and both poles, needle-like and tile-covering Gaussians, a last ragged tile row)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, GRAD_TOL, IMG_TOL, oracle_settings, rel_l2, to_torch

pytestmark = pytest.mark.gpu
W, H = 128, 59


def _scene():
    sc = S.random_scene(900, W, H, seed=311, sh_degree=1, log_scale=(-2.8, 0.9))
    rng = np.random.default_rng(311)
    m = sc.means
    m[:120] = np.stack([0.05 * rng.normal(size=120), rng.uniform(-1, 1, 120), -2 + 0.1 * rng.normal(size=120)], 1)
    m[120:240] = np.stack([0.15 * rng.normal(size=120), np.sign(rng.normal(size=120)) * 2.0, 0.15 * rng.normal(size=120)], 1)
    sc.scales[240:300, 0] *= 20.0  # needles and discs several tiles long
    sc.scales[240:300, 1:] *= 0.05
    return sc


def _run(sc, **kw):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    rast = Rasterizer()
    rs = RenderSettings(sh_degree=1, **kw)
    imgs, Ts = rast.forward(*to_torch(sc), sc.views, rs)
    w = np.random.default_rng(5).normal(size=(3, H, W)).astype(np.float32)
    g = rast.backward([torch.tensor(w, device="cuda")])
    torch.cuda.synchronize()
    assert rast.status() == 0
    return imgs[0].cpu().numpy(), Ts[0].cpu().numpy(), {k: g[k].cpu().numpy().astype(np.float64) for k in GRAD_NAMES}


# regions of 4, 8, 16 columns x 8 rows; tile heights that no region of 8 rows divides (whole tile rows);
# eight pixels per thread; the automatic choice
LAYOUTS = [(16, 16, 1, 1), (16, 16, 2, 2), (16, 16, 4, 4), (16, 16, 8, 8), (32, 8, 1, 2), (32, 16, 4, 8), (8, 32, 1, 1),
           (8, 16, 2, 4), (16, 6, 1, 1), (8, 12, 1, 1), (32, 4, 2, 1), (16, 16, 0, 0), (32, 32, 0, 0)]


@pytest.fixture(scope="module")
def base():
    sc = _scene()
    img, T, g = _run(sc, pixels_per_thread=2, pixels_per_thread_bwd=4)
    return sc, img, T, g


@pytest.mark.parametrize("tw,th,ppt,ppt_bwd", LAYOUTS)
def test_layouts_agree(base, tw, th, ppt, ppt_bwd):
    sc, img, T, g = base
    i2, T2, g2 = _run(sc, tile_w=tw, tile_h=th, pixels_per_thread=ppt, pixels_per_thread_bwd=ppt_bwd)
    assert np.array_equal(i2, img) and np.array_equal(T2, T)
    # the same contributions in another order: the suite's gradient tolerance bounds the rounding of
    # float32 sums that cancel (needle-like Gaussians under random weights)
    for k in GRAD_NAMES:
        assert rel_l2(g2[k], g[k]) <= GRAD_TOL, k


def test_lists_and_walk_lose_no_entry(base):
    """Forward against the oracle, which tests every Gaussian at every pixel."""
    sc, img, _, _ = base
    from paper_2410_20686_gb300.rasterizer import RenderSettings
    ref, _, _, margins = O.render(O.Params.of(sc), sc.views[0], oracle_settings(RenderSettings(sh_degree=1)))
    ok = ~O.ambiguous(margins)
    assert np.abs(img - ref).max(axis=0)[ok].max() <= IMG_TOL
