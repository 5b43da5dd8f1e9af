"""Which frames partition their items (three launches more): those of two perspective views and more, at least
as many as ERP views, and 2^17 items; and their images and gradients are the single views' either way."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("faces,erp,partitioned", [(1, 0, False), (2, 0, True), (1, 1, False), (1, 3, False), (2, 1, True),
                                                   (2, 2, True), (2, 3, False)])
def test_rule(faces, erp, partitioned):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    at, nv = (0.1, 0.0, -0.2), faces + erp
    views = S.cubemap_views(64, at)[:faces] + [S.yaw_view(64, 64, at, 0.7 * k) for k in range(erp)]
    n = -(-(1 << 17) // nv)
    sc = S.random_scene(n, 64, 64, seed=60 + nv, sh_degree=1, radius=(0.1, 5.0), log_scale=(-4.5, 0.5))
    p, rs = to_torch(sc), RenderSettings(sh_degree=1)
    w = [torch.randn(3, 64, 64, device="cuda", generator=torch.Generator("cuda").manual_seed(k)) for k in range(nv)]

    def run(vs, ws, count=n):
        r = Rasterizer(capacity_mode="fixed")
        r.reserve_pairs(1 << 22)
        imgs, _ = r.forward(*[t[:count].contiguous() for t in p], vs, rs)
        launches = r.launch_count()
        g = r.backward(ws)
        assert r.status() == 0
        return imgs, {k: v.cpu().numpy().astype(np.float64) for k, v in g.items()}, launches

    imgs, grads, launches = run(views, w)
    fewer = run(views, w, n - 1)[2]  # below 2^17 items
    assert launches - fewer == (3 if partitioned else 0)
    sums = None
    for k in range(nv):
        one, g, _ = run([views[k]], [w[k]])
        assert torch.equal(imgs[k], one[0]), k
        sums = g if sums is None else {name: sums[name] + g[name] for name in g}
    for name in GRAD_NAMES:  # the same terms: only the order of the additions differs
        assert rel_l2(grads[name], sums[name]) < 1e-5, name
