"""The backward preprocess with its SH rows staged through shared memory (degrees 1 and 3 without
coefficients above the degree) against the same frame with one unused coefficient more, which takes the
path of one thread per row: counts around a warp and a CTA, one and several views, written and added."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg", [1, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 1000])
@pytest.mark.parametrize("views,accumulate", [(1, False), (1, True), (3, False), (3, True)])
def test_staged_rows_match_unstaged(deg, n, views, accumulate):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(n, 64, 32, seed=500 + n, sh_degree=deg, log_scale=(-1.8, 0.5))
    sc.sh[: n // 3, 0] = -2.0  # clamped channels
    vs = [S.yaw_view(64, 32, (0.2 * k, 0.0, 0.1), 0.9 * k) for k in range(views)]
    rng = np.random.default_rng(n)
    w = [torch.tensor(rng.normal(size=(3, 32, 64)), dtype=torch.float32, device="cuda") for _ in vs]
    out = []
    for pad in (0, 1):
        p = to_torch(sc)
        p[4] = torch.cat([p[4], torch.full((n, pad, 3), 7.0, device="cuda")], dim=1).contiguous()
        rast = Rasterizer()
        rast.forward(*p, vs, RenderSettings(sh_degree=deg, grad_accumulate=accumulate))
        grads = {k: torch.full_like(t, 0.5) for k, t in zip(GRAD_NAMES, p)}
        rast.backward(w, grads)
        torch.cuda.synchronize()
        assert rast.status() == 0
        out.append({k: t.cpu().numpy().astype(np.float64) for k, t in grads.items()})
    k = (deg + 1) ** 2
    assert np.all(out[1]["sh"][:, k:] == (0.5 if accumulate else 0.0))
    out[1]["sh"] = out[1]["sh"][:, :k]
    for name in GRAD_NAMES:  # the same sums but for the order of the blend's atomic additions
        assert rel_l2(out[0][name], out[1][name]) < 1e-5, name
