"""The streaming D-SSIM passes at the edges of their strips (64 columns), segments and row ring, on
odd widths (padded map rows, unpaired last columns) and images smaller than the window."""
import numpy as np
import pytest

from oracle import loss as OL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,wrap", [(64, 8, True), (65, 33, True), (63, 17, False), (129, 75, False), (128, 3, True),
                                      (7, 40, True), (11, 5, False), (1, 1, False), (200, 301, True), (1999, 121, True)])
@pytest.mark.parametrize("shift", [0, 1])
def test_strips_match_the_oracle(W, H, wrap, shift):
    import torch
    from paper_2410_20686_gb300.loss import l1_dssim
    rng = np.random.default_rng(W * 1000 + H)
    y = rng.uniform(size=(3, H, W)).astype(np.float32)
    x = np.clip(y + rng.normal(scale=0.1, size=y.shape), 0, 1).astype(np.float32)

    def put(a):  # contiguous, `shift` floats past a 16-byte boundary
        t = torch.zeros(a.size + 8, device="cuda")[shift:shift + a.size].view(a.shape)
        return t.copy_(torch.from_numpy(a))

    loss, grads = l1_dssim([put(x)], [put(y)], wrap_u=wrap)
    alone, none = l1_dssim([put(x)], [put(y)], wrap_u=wrap, want_grad=False)
    assert float(alone) == float(loss) and none == [None]
    ref_loss, ref_grad = OL.loss_and_grad(x, y, wrap_u=wrap)
    # float32 storage of the moments and a fixed-order float32 sum, as in the suite's other loss tests
    assert float(loss) == pytest.approx(ref_loss, rel=1e-5)
    g = grads[0].cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - ref_grad) <= 1e-4 * np.linalg.norm(ref_grad)
    np.testing.assert_allclose(g, ref_grad, rtol=0, atol=1e-4 * np.abs(ref_grad).max())
