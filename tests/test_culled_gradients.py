"""Gradients of frames that partition their items: the backward preprocess takes only the views that do not
cull a Gaussian. Against the single views' gradients and statistics (each view alone has too few items for the
partition), with SH rows staged and not, and for Gaussians seen by no view, by one, and by all of them."""
from types import SimpleNamespace

import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg,pad", [(0, 0), (1, 0), (2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("kind", ["cube", "mixed", "64 views"])
def test_gradients_match_single_views(deg, pad, kind):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    n = {"cube": 21_857, "mixed": 43_711, "64 views": 2_063}[kind]
    sc = S.random_scene(n, 64, 64, seed=70 + deg, sh_degree=deg, radius=(0.1, 5.0), log_scale=(-4.5, 0.5))
    sc.sh[: n // 3, 0] = -2.0  # clamped channels
    sc.opacity[::7] = 0.001  # below 1 / 255: culled everywhere
    faces = S.cubemap_views(64, (0.1, 0.0, -0.2))
    views = {"cube": faces, "mixed": [faces[1], S.yaw_view(96, 48, (0.1, 0.0, -0.2), 0.3), faces[4]],
             "64 views": (faces * 11)[:64]}[kind]
    p = to_torch(sc)
    p[4] = torch.cat([p[4], torch.full((n, pad, 3), 7.0, device="cuda")], dim=1).contiguous()
    gen = torch.Generator("cuda").manual_seed(deg)
    w = [torch.randn(3, v.height, v.width, device="cuda", generator=gen) for v in views]

    def run(vs, ws):
        st = SimpleNamespace(grad=torch.zeros(n, device="cuda"), elev=torch.zeros(n, device="cuda"),
                             count=torch.zeros(n, dtype=torch.int32, device="cuda"))
        r = Rasterizer()
        r.forward(*p, vs, RenderSettings(sh_degree=deg))
        g = {k: v.double() for k, v in r.backward(ws, densify=st).items()}
        assert r.status() == 0
        return g, st

    got, stats = run(views, w)
    sums, counts = None, torch.zeros(n, dtype=torch.int32, device="cuda")
    grad, elev = torch.zeros(n, device="cuda", dtype=torch.float64), torch.zeros(n, device="cuda", dtype=torch.float64)
    for v, wv in zip(views, w):
        g, st = run([v], [wv])
        sums = g if sums is None else {k: sums[k] + g[k] for k in g}
        grad, elev, counts = grad + st.grad.double(), elev + st.elev.double(), counts + st.count
    assert torch.equal(stats.count, counts) and int((counts == 0).sum()) > 0
    assert rel_l2(stats.grad.double().cpu().numpy(), grad.cpu().numpy()) < 1e-5
    assert rel_l2(stats.elev.double().cpu().numpy(), elev.cpu().numpy()) < 1e-5
    for name in GRAD_NAMES:  # the same terms: only the order of the additions differs
        assert rel_l2(got[name].cpu().numpy(), sums[name].cpu().numpy()) < 1e-5, name
