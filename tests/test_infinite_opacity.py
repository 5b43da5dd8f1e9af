"""An infinite opacity blends as any very large one does, and counts as it does: a pixel that has stopped, or lies
below the image, takes no part in its entries."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ppt", [1, 2, 4])
def test_counts_as_a_very_large_one(ppt):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(60, 64, 36, seed=8, sh_degree=0, radius=(1.0, 3.0), log_scale=(1.5, 0.2))  # four rows in the last tiles
    sc.opacity[:] = 0.9
    rs = RenderSettings(sh_degree=0, full_lists=True, pixels_per_thread=ppt)
    out = []
    for value in (1e30, np.inf):
        sc.opacity[::2] = value
        r = Rasterizer()
        (img,), (T,) = r.forward(*to_torch(sc), sc.views, rs)
        out.append((img, T, r.stats()))
    (img, T, st), (inf_img, inf_T, inf_st) = out
    assert inf_st["pairs"] == st["pairs"] == 60 * 4 * 3  # every footprint meets every tile
    assert torch.equal(img, inf_img) and torch.equal(T, inf_T)
    assert all(inf_st[k] == st[k] for k in ("evals_fwd", "blended", "entries_tile"))
