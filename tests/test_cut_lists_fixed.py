"""Cut lists of frames of few pairs. A host that knows of at most 32768 pairs keeps the whole lists, so these frames
are rendered in fixed mode, as a captured step is: the emission's compaction around its limits for every tile shape
against the whole lists, and an image and its final T against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, compare_image, oracle_settings, rel_l2, to_torch

pytestmark = pytest.mark.gpu


def _rast():
    from paper_2410_20686_gb300.rasterizer import Rasterizer
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(1 << 20)
    return r


def _scene(n_near, n_far, width, height, seed, near=0.0):
    """Large opaque Gaussians on one side of many small ones, some across the seam: tiles saturate on that side."""
    sc = S.random_scene(n_near + n_far, width, height, seed=seed, sh_degree=1, radius=(3.0, 8.0), log_scale=(-2.4, 0.7))
    d = np.random.default_rng(seed).normal(size=(n_near, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    d[:, 0] = np.abs(d[:, 0])
    d[: n_near // 8, 2] = -np.abs(d[: n_near // 8, 2])
    sc.means[:n_near] = (1.3 * d).astype(np.float32)
    sc.scales[:n_near] = np.float32(np.exp(near))
    sc.opacity[:n_near] = 0.97
    return sc


@pytest.mark.parametrize("tile", [(8, 4), (8, 8), (8, 16), (16, 16), (32, 8), (32, 32)])
def test_every_shape(tile):
    import torch
    from paper_2410_20686_gb300.rasterizer import RenderSettings
    sc = _scene(40, 3000, 512, 256, 61)
    p, kw = to_torch(sc), dict(sh_degree=1, tile_w=tile[0], tile_h=tile[1])
    w = [torch.randn(3, 256, 512, device="cuda", generator=torch.Generator("cuda").manual_seed(2))]
    out = []
    for full in (True, False):
        r = _rast()
        (img,), (T,) = r.forward(*p, sc.views, RenderSettings(full_lists=full, **kw))
        g = r.backward(w)
        assert r.status() == 0
        out.append((img, T, g, r.stats(), r.debug_lists()))
    (img, T, g, st, whole), (cimg, cT, cg, cst, cut) = out
    assert st["pairs_sorted"] == st["pairs"] == cst["pairs"] > 1.05 * cst["pairs_sorted"]
    assert torch.equal(img, cimg) and torch.equal(T, cT)
    for a, b in zip(whole["ranges"], cut["ranges"]):  # every cut list is a prefix of the whole one
        k = int(b[1] - b[0])
        assert np.array_equal(cut["pair_items"][b[0]:b[1]], whole["pair_items"][a[0]:a[0] + k])
    for name in GRAD_NAMES:  # the same terms: only the order of the additions differs
        assert rel_l2(cg[name].cpu().numpy(), g[name].cpu().numpy()) < 1e-5, name


def test_against_the_oracle():
    import torch
    from paper_2410_20686_gb300.rasterizer import RenderSettings
    sc = _scene(40, 400, 128, 64, 62, near=0.2)
    rs, r = RenderSettings(sh_degree=1, bg=(0.2, 0.5, 0.1), tile_w=8, tile_h=8), _rast()
    (img,), (T,) = r.forward(*to_torch(sc), sc.views, rs)
    torch.cuda.synchronize()
    st = r.stats()
    assert st["status"] == 0 and st["pairs_sorted"] < st["pairs"] <= 32768
    ref, Tref, _, margins = O.render(O.Params.of(sc), sc.views[0], oracle_settings(rs))
    compare_image(img.cpu().numpy().astype(np.float64), ref, margins)
    amb = O.ambiguous(margins, 2e-5, 1e-4)
    assert np.abs(T.cpu().numpy() - Tref)[~amb].max() <= 1e-4
