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


@pytest.mark.parametrize("floats", [1216, 1217, 5000, 8192, 20000])
def test_partial_sums_fit_the_scratch(floats):
    """Through the C entry: the least scratch there is takes fewer CTAs, and nothing past its end is written."""
    import ctypes as C

    import torch
    from paper_2410_20686_gb300 import _lib as L
    g = torch.Generator("cuda").manual_seed(4)
    x, y = (torch.rand(3, 4096, 2048, device="cuda", generator=g) for _ in range(2))
    grad, loss, scratch = torch.empty_like(x), torch.empty(1, device="cuda"), torch.full((floats + 64,), -7.0, device="cuda")
    ptr, one = C.c_void_p * 1, C.c_int * 1

    def call(nbytes):
        return L.load().odgs_loss_l1(ptr(x.data_ptr()), ptr(y.data_ptr()), one(2048), one(4096), 1,
                                     C.byref(L.LossParams(0.0, 0, 0, 0)), ptr(grad.data_ptr()), C.c_void_p(loss.data_ptr()),
                                     C.c_void_p(scratch.data_ptr()), C.c_size_t(nbytes), L.raw_stream(x.device))

    assert call(1216 * 4 - 4) == L.ODGS_ERR_WORKSPACE
    assert call(4 * floats) == L.ODGS_OK
    assert bool((scratch[floats:] == -7.0).all())
    assert float(loss) == pytest.approx(float((x.double() - y.double()).abs().mean()), rel=1e-5)
    assert torch.equal(grad, (x - y).sign() / x.numel())
