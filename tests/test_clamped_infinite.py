"""Colour channels clamped by an infinite coefficient: their colour is 0 and they carry no gradient, as
with any other negative colour, in frames of one view and of several, with SH rows staged and not."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg,pad", [(1, 0), (2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("n_views", [1, 2, 6])
def test_infinite_coefficient_clamps_as_any_negative_colour(deg, pad, n_views):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    n = 22_000 if n_views == 6 else 700  # six perspective views of 22K: items partitioned
    sc = S.random_scene(n, 64, 64, seed=90 + deg, sh_degree=deg, radius=(0.5, 4.0), log_scale=(-3.0, 0.5))
    at = (0.1, 0.0, -0.2)
    views = S.cubemap_views(64, at) if n_views == 6 else [S.yaw_view(64, 64, at, 0.4 * k) for k in range(n_views)]
    p = to_torch(sc)
    # the first coefficient of degree 1 is that of y: its channel is clamped in every view
    y = p[0][:, 1]
    side = torch.where(y.abs() > 0.5, y.sign(), torch.zeros_like(y))
    side[1::2] = 0.0
    assert int((side != 0).sum()) > 50
    p[4] = torch.cat([p[4], torch.zeros(n, pad, 3, device="cuda")], dim=1).contiguous()
    w = [torch.randn(3, 64, 64, device="cuda", generator=torch.Generator("cuda").manual_seed(k)) for k in range(n_views)]

    def run(value):
        p[4][side > 0, 1, 1], p[4][side < 0, 1, 1] = -value, value
        r = Rasterizer()
        imgs, _ = r.forward(*p, views, RenderSettings(sh_degree=deg))
        g = r.backward(w)
        assert r.status() == 0
        return imgs, {k: v.cpu().numpy().astype(np.float64) for k, v in g.items()}

    images, want = run(1e4)
    inf_images, got = run(float("inf"))
    assert all(torch.equal(a, b) for a, b in zip(images, inf_images))
    for name in GRAD_NAMES:  # the same terms: only the order of the additions differs
        assert np.isfinite(got[name]).all() and rel_l2(got[name], want[name]) < 1e-5, name
