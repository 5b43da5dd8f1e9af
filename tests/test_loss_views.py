"""The L1 term of many views in one pass: each view's gradient is the single view's bit for bit, and the
loss the oracle's sum, over sizes with and without whole 16-byte rows and more views than one launch holds."""
import numpy as np
import pytest

from oracle import loss as OL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,area", [([(256, 128), (64, 32), (37, 21), (2048, 3)], True), ([(1, 1), (5, 700), (128, 1)], False),
                                        ([(16 + k, 8 + k % 5) for k in range(70)], True)])
@pytest.mark.parametrize("want_grad", [True, False])
def test_views_in_one_pass(sizes, area, want_grad):
    import torch
    from paper_2410_20686_gb300.loss import l1_dssim
    rng = np.random.default_rng(len(sizes))
    xs = [rng.uniform(size=(3, h, w)).astype(np.float32) for w, h in sizes]
    ys = [rng.uniform(size=(3, h, w)).astype(np.float32) for w, h in sizes]
    for x, y in zip(xs, ys):
        x[0, 0, 0] = y[0, 0, 0]  # gradient 0 where they are equal
    X, Y = ([torch.from_numpy(a).cuda() for a in t] for t in (xs, ys))
    loss, grads = l1_dssim(X, Y, lam=0.0, area_weight=area, want_grad=want_grad)
    want = 0.0
    for k, (x, y) in enumerate(zip(xs, ys)):
        ref, ref_grad = OL.loss_and_grad(x, y, lam=0.0, area_weight=area, wrap_u=False)  # no window: any wrap
        want += ref
        if not want_grad:
            assert grads[k] is None
            continue
        one = l1_dssim([X[k]], [Y[k]], lam=0.0, area_weight=area)[1][0]
        assert torch.equal(grads[k], one)
        np.testing.assert_allclose(grads[k].cpu().numpy(), ref_grad, rtol=0, atol=1e-4 * np.abs(ref_grad).max())
    assert float(loss) == pytest.approx(want, rel=1e-5)
