"""The depth sort around its tiles and the look-back's groups of four tiles: the order is that of a stable
sort, for counts next to multiples of a tile (2048 items, 4096 from 2^20 items on), equal keys, few and many
digits, and with the look-back's words read in any state of their tiles."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 4096, 4097, 8193, 10_239, 10_241, 18_431, 200_001,
                               (1 << 20) - 1, 1 << 20, (1 << 20) + 5 * 4096 + 1])
@pytest.mark.parametrize("depths", ["random", "equal", "two"])
def test_depth_order(n, depths):
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    g = torch.Generator("cuda").manual_seed(n)
    d = torch.randn(n, 3, device="cuda", generator=g)
    d = d / d.norm(dim=1, keepdim=True)
    odd = (torch.arange(n, device="cuda") % 2).float()[:, None]
    means = {"random": lambda: d * (torch.rand(n, 1, device="cuda", generator=g) * 5.0 + 0.2),
             "equal": lambda: d[:1] * 2.0 + 0.0 * odd, "two": lambda: d[:1] * (1.0 + odd)}[depths]().contiguous()
    sc = S.random_scene(1, 64, 32, seed=1, sh_degree=0, log_scale=(-4.5, 0.1))
    rest = [t[:1].expand(n, *t.shape[1:]).contiguous() for t in to_torch(sc)[1:]]
    rest[0].fill_(1e-3)
    rast = Rasterizer()
    for _ in range(2):
        rast.forward(means, *rest, [S.yaw_view(64, 32, (0.0, 0.0, 0.0), 0.0)], RenderSettings(sh_degree=0))
        assert rast.status() == 0
        out = rast.debug_lists()
        k, i = out["depth_keys"].astype(np.uint64), out["depth_items"].astype(np.uint64)
        assert np.array_equal(np.sort(i), np.arange(n, dtype=np.uint64))
        words = (k << np.uint64(32)) | i
        assert np.all(words[1:] > words[:-1])
        assert len(np.unique(k)) <= {"random": n, "equal": 1, "two": 2}[depths]
