"""Perspective frames of many items test all views of a Gaussian cheaply before they project it: nothing that
the projection keeps is culled. Images, visible items and pairs are those of the single views (too few items
for that path), bit for bit, for principal points off the centre and outside the image, unequal
focal lengths, cameras far from the origin, centres along the 30 % border, and Gaussians behind the camera."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


def _views(kind, shift):
    fx, fy, cx, cy = {"plain": (48.0, 48.0, 48.0, 32.0), "off": (20.0, 90.0, 5.0, 60.0), "out": (60.0, 35.0, -70.0, 150.0)}[kind]
    out = []
    for k in range(5):
        a, b = 1.3 * k, 0.7 * k
        ry = np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]])
        rx = np.array([[1, 0, 0], [0, np.cos(b), -np.sin(b)], [0, np.sin(b), np.cos(b)]])
        R = rx @ ry
        c = np.array([0.1 * k, -0.2, 0.3]) + shift
        out.append(S.pinhole_view(96, 64, fx, fy, cx=cx, cy=cy, R_wc=R, t_wc=-R @ c))
    return out


@pytest.mark.parametrize("shift", [0.0, 3000.0])
@pytest.mark.parametrize("kind", ["plain", "off", "out"])
def test_frame_matches_single_views(kind, shift):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    n = 27_000  # five views: 135000 items
    sc = S.random_scene(n, 64, 64, seed=11, sh_degree=1, radius=(0.05, 6.0), log_scale=(-4.0, 0.8))
    p = to_torch(sc)
    views = _views(kind, shift)
    v0 = views[0]  # centres on and next to the border that the cull draws
    u = torch.tensor([-0.3, 1.3], device="cuda")[torch.arange(2000, device="cuda") % 2] * v0.width
    z = torch.rand(2000, device="cuda") + 0.5
    fx, cx = {"plain": (48.0, 48.0), "off": (20.0, 5.0), "out": (60.0, -70.0)}[kind]
    t = torch.stack([(u - cx) / fx * z, torch.zeros_like(z), z], 1).double()
    R = torch.tensor(np.asarray(v0.R_wc), device="cuda").double()
    p[0] += shift
    p[0][:2000] = ((t - torch.tensor(np.asarray(v0.t_wc), device="cuda").double()) @ R).float()
    rs = RenderSettings(sh_degree=1)
    r = Rasterizer()
    imgs, _ = r.forward(*p, views, rs)
    st = r.stats()
    assert st["status"] == 0
    visible = pairs = 0
    for img, v in zip(imgs, views):
        one = Rasterizer()
        (ref,), _ = one.forward(*p, [v], rs)
        assert torch.equal(img, ref)
        s1 = one.stats()
        visible, pairs = visible + s1["visible"], pairs + s1["pairs"]
    assert (st["visible"], st["pairs"]) == (visible, pairs)


def test_sort_that_gives_up_reads_no_stale_record():
    """A frame whose sorts give up at once (a wait limit of 0), on a workspace of NaN bytes and a pair buffer
    that lists items which this frame culls: flagged, with finite images and gradients, then exact again."""
    import torch
    from paper_2410_20686_gb300 import _lib as L
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(30_000, 96, 96, seed=5, sh_degree=1, radius=(0.3, 5.0), log_scale=(-3.5, 0.6))
    p, rs, views = to_torch(sc), RenderSettings(sh_degree=1), S.cubemap_views(96, (0.1, 0.0, -0.2))
    turned = [views[k] for k in (1, 0, 3, 2, 5, 4)]
    r = Rasterizer()
    r.reserve_pairs(4 << 20)
    r.forward(*p, turned, rs)
    torch.cuda.synchronize()
    r.ws.fill_(255)
    r.set_wait_limit(0)
    imgs, _ = r.forward(*p, views, rs)
    g = r.backward([torch.ones_like(i) for i in imgs])
    torch.cuda.synchronize()
    assert r.status() & L.DEV_TIMEOUT
    assert all(torch.isfinite(i).all() for i in imgs) and all(torch.isfinite(t).all() for t in g.values())
    r.set_wait_limit(1 << 22)
    imgs, _ = r.forward(*p, views, rs)
    ref, _ = Rasterizer().forward(*p, views, rs)
    assert r.status() == 0 and all(torch.equal(a, b) for a, b in zip(imgs, ref))
