"""A captured frame replayed on a context that has rendered an eager frame in between: what follows the replay
(lists rebuilt for the backward pass, its gradients) follows the replayed frame, not the host's last call."""
import numpy as np
import pytest

from paper_2410_20686_gb300 import scenes as S
from helpers import GRAD_NAMES, rel_l2, to_torch

pytestmark = pytest.mark.gpu


def _scene(n=200, seed=41):
    """Few pairs, and tiles that saturate early in their lists."""
    sc = S.random_scene(n, 256, 128, seed=seed, sh_degree=0, radius=(1.0, 3.0), log_scale=(0.5, 0.2))
    sc.opacity[:] = 0.98
    return sc


def _capture(r, p, views, rs):
    import torch
    r.capacity_mode = "fixed"
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.preprocess(*p, views, rs)
        r.bin_sort()
        imgs, _ = r.render_fwd(want_T=False)
    return g, imgs


def _upstream(views):
    import torch
    return [torch.randn(3, v.height, v.width, device="cuda", generator=torch.Generator("cuda").manual_seed(k))
            for k, v in enumerate(views)]


def _check_grads(got, want):
    for name in GRAD_NAMES:  # the same terms: only the order of the additions differs
        assert rel_l2(got[name].cpu().numpy().astype(np.float64), want[name].cpu().numpy().astype(np.float64)) < 1e-5, name


def test_rebuild_after_a_replay_and_an_eager_frame_of_few_pairs():
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = _scene()
    p, w = to_torch(sc), _upstream(sc.views)
    rs = RenderSettings(sh_degree=0, recompute_lists=True)
    ref = Rasterizer(capacity_mode="fixed")  # pairs unknown to the host: cut lists
    ref.reserve_pairs(1 << 17)
    want_imgs, _ = ref.forward(*p, sc.views, rs)
    want, lists = ref.backward(w), ref.debug_lists()
    st = ref.stats()
    assert st["pairs_sorted"] < 0.8 * st["pairs"] and st["pairs"] <= 32768
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(1 << 17)
    r.forward(*p, sc.views, rs)
    graph, imgs = _capture(r, p, sc.views, rs)
    for _ in range(2):
        r.capacity_mode = "query"
        r.forward(*p, sc.views, rs)  # its pairs are known: whole lists
        assert r.stats()["pairs_sorted"] in (st["pairs"], st["pairs_sorted"])
        r.capacity_mode = "fixed"
        graph.replay()
        assert r.stats()["pairs_sorted"] == st["pairs_sorted"] and torch.equal(imgs[0], want_imgs[0])
        got = r.backward(w)
        d = r.debug_lists()
        assert r.status() == 0
        for key in ("pair_tiles", "pair_items", "ranges"):
            k = st["pairs_sorted"] if key != "ranges" else None
            assert np.array_equal(d[key][:k], lists[key][:k]), key
        _check_grads(got, want)


@pytest.mark.parametrize("rebuild", [False, True])
@pytest.mark.parametrize("first", ["erp", "perspective"])
def test_backward_after_a_replay_and_an_eager_frame_of_another_camera(first, rebuild):
    """Frames of perspective views sort their visible items alone; the others all items."""
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    n, at = 22_000, (0.1, 0.0, -0.2)
    sc = S.random_scene(n, 64, 64, seed=43, sh_degree=1, radius=(0.1, 5.0), log_scale=(-4.0, 0.5))
    sc.opacity[::5] = 0.001  # below 1 / 255: culled in every view
    kinds = {"perspective": S.cubemap_views(64, at), "erp": [S.yaw_view(64, 64, at, 0.7 * k) for k in range(6)]}
    views = kinds.pop(first)
    (other,) = kinds.values()
    p, w = to_torch(sc), _upstream(views)
    rs = RenderSettings(sh_degree=1, recompute_lists=rebuild)
    ref = Rasterizer(capacity_mode="fixed")
    ref.reserve_pairs(1 << 21)
    want_imgs, _ = ref.forward(*p, views, rs)
    want = ref.backward(w)
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(1 << 21)
    r.forward(*p, views, rs)
    graph, imgs = _capture(r, p, views, rs)
    r.forward(*p, other, rs)
    r.backward(w)
    graph.replay()
    got = r.backward(w)
    assert r.status() == 0 and all(torch.equal(a, b) for a, b in zip(imgs, want_imgs))
    _check_grads(got, want)
    alone = torch.cuda.CUDAGraph()
    with torch.cuda.graph(alone):
        r.preprocess(*p, views, rs)
    r.forward(*p, other, rs)
    alone.replay()  # the projection alone: the binning is the host's
    r.bin_sort()
    imgs, _ = r.render_fwd(want_T=False)
    got = r.backward(w)
    assert r.status() == 0 and all(torch.equal(a, b) for a, b in zip(imgs, want_imgs))
    _check_grads(got, want)


def _pairs(r, name):
    import ctypes as C
    from paper_2410_20686_gb300 import _lib as L
    k = C.c_size_t()
    assert getattr(r.lib, name)(r.ctx, C.byref(k), L.raw_stream(r.device)) == L.ODGS_OK
    return int(k.value)


def test_pair_count_after_a_replay_that_brings_more_pairs():
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = _scene()
    p, rs = to_torch(sc), RenderSettings(sh_degree=0)
    scales = p[1].clone()
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(1 << 17)
    r.forward(*p, sc.views, rs)
    many = _pairs(r, "odgs_query_pairs")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.preprocess(*p, sc.views, rs)
    for _ in range(2):
        p[1].copy_(0.05 * scales)
        r.preprocess(*p, sc.views, rs)
        few = _pairs(r, "odgs_wait_pairs")  # makes the event, or is the second eager frame
        p[1].copy_(scales)
        torch.cuda._sleep(20_000_000)  # the replay is still to come when the count is asked for
        g.replay()
        assert _pairs(r, "odgs_wait_pairs") == many > 4 * few


def test_binning_captured_after_a_query_takes_any_number_of_pairs():
    import torch
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = _scene()
    p, rs = to_torch(sc), RenderSettings(sh_degree=0)
    ref = Rasterizer(capacity_mode="fixed")
    ref.reserve_pairs(1 << 17)
    (want,), _ = ref.forward(*p, sc.views, rs)
    st = ref.stats()
    cap = (st["pairs"] + st["pairs_sorted"]) // 2  # the cut lists fit, the whole ones do not
    assert st["pairs_sorted"] < cap < st["pairs"]
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(cap)
    scales = p[1].clone()
    p[1].copy_(0.05 * scales)
    r.forward(*p, sc.views, rs)
    assert r.query_pairs() < cap
    r.preprocess(*p, sc.views, rs)
    r.query_pairs()  # few pairs, which would fit
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.bin_sort()
        (img,), _ = r.render_fwd(want_T=False)
    p[1].copy_(scales)
    r.preprocess(*p, sc.views, rs)
    g.replay()
    assert r.status() == 0 and r.stats()["pairs_sorted"] <= cap
    assert torch.equal(img, want)


def test_launches_of_a_graphed_frame_are_the_replayed_ones():
    import torch
    from paper_2410_20686_gb300.graph import GraphedFrame
    from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings
    sc = _scene()  # few pairs: the sizing run keeps whole lists, the captured step cuts them
    p, rs = to_torch(sc), RenderSettings(sh_degree=0)
    frame = GraphedFrame(p, sc.views, [torch.rand(3, 128, 256, device="cuda")], rs)
    r = Rasterizer(capacity_mode="fixed")
    r.reserve_pairs(1 << 17)
    r.forward(*p, sc.views, rs)
    r.backward(_upstream(sc.views))
    assert frame.launches == r.launch_count()
