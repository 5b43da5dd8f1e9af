"""The L1 pass around its number of CTAs (8192 rows of three channels): fewer rows, as many, one more and several
times as many, in one view and in several, against the oracle."""
import numpy as np
import pytest

from oracle import loss as OL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heights", [(2730,), (2731,), (2000, 731), (5462, 3), (16384,)])
def test_rows_around_the_ctas(heights):
    import torch
    from paper_2410_20686_gb300.loss import l1_dssim
    rng = np.random.default_rng(len(heights) + heights[0])
    xs, ys = ([rng.uniform(size=(3, h, 8)).astype(np.float32) for h in heights] for _ in range(2))
    loss, grads = l1_dssim([torch.from_numpy(x).cuda() for x in xs], [torch.from_numpy(y).cuda() for y in ys], lam=0.0)
    want = 0.0
    for x, y, g in zip(xs, ys, grads):
        ref, ref_grad = OL.loss_and_grad(x, y, lam=0.0, area_weight=True, wrap_u=False)
        want += ref
        np.testing.assert_allclose(g.cpu().numpy(), ref_grad, rtol=0, atol=1e-4 * np.abs(ref_grad).max())
    assert float(loss) == pytest.approx(want, rel=1e-5)
