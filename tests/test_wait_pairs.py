"""odgs_wait_pairs: the count of odgs_query_pairs at every stage of a frame, after a captured preprocess,
and on an empty scene; a frame that uses it equals one that synchronizes."""
import ctypes as C

import numpy as np
import pytest

from paper_2410_20686_gb300 import _lib as L
from paper_2410_20686_gb300 import scenes as S
from helpers import to_torch

pytestmark = pytest.mark.gpu


def _call(r, name):
    p = C.c_size_t()
    st = getattr(r.lib, name)(r.ctx, C.byref(p), L.raw_stream(r.device))
    return st, int(p.value)


def test_counts_agree_at_every_stage():
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    rs = RenderSettings(sh_degree=2)
    r = Rasterizer()
    assert _call(r, "odgs_wait_pairs")[0] == L.ODGS_ERR_STATE
    want = None
    for k in range(4):  # the first call of a context, then the recorded projections
        sc = S.random_scene(5000 + 1000 * k, 256, 128, seed=70 + k, sh_degree=2)
        p = to_torch(sc)
        r.preprocess(*p, sc.views, rs)
        first = _call(r, "odgs_wait_pairs")
        want = _call(r, "odgs_query_pairs")
        assert first == want and want[0] == L.ODGS_OK and want[1] > 0
        r.reserve_pairs(want[1])
        r.bin_sort()
        assert _call(r, "odgs_wait_pairs") == want  # later stages
        (img,), _ = r.render_fwd(want_T=False)
        assert _call(r, "odgs_wait_pairs") == want
    r.capacity_mode = "fixed"
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.preprocess(*p, sc.views, rs)
        r.bin_sort()
        r.render_fwd(images=[img], want_T=False)
    ref = img.clone()
    g.replay()
    torch.cuda.synchronize()
    assert _call(r, "odgs_wait_pairs") == want and torch.equal(img, ref)
    r.preprocess(*p, sc.views, rs)  # eager again
    assert _call(r, "odgs_wait_pairs") == want


def test_overflow_and_empty_scene():
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = S.random_scene(3000, 256, 128, seed=77, sh_degree=0)
    p, rs = to_torch(sc), RenderSettings(sh_degree=0, full_lists=True)
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(64)
    for _ in range(2):
        r.preprocess(*p, sc.views, rs)
        r.bin_sort()
        assert _call(r, "odgs_wait_pairs")[0] == L.ODGS_ERR_CAPACITY
    empty = [t[:0].contiguous() for t in p]
    for _ in range(2):
        r.preprocess(*empty, sc.views, rs)
        assert _call(r, "odgs_wait_pairs") == (L.ODGS_OK, 0)
        r.bin_sort()
        (img,), _ = r.render_fwd(want_T=False)
        torch.cuda.synchronize()
        assert np.array_equal(img.cpu().numpy(), np.zeros((3, 128, 256), np.float32))
