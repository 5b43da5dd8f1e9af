"""The densification kernels at the edges of their groups (256 slots, four Gaussians a thread), on SH rows
that are no multiple of 16 bytes and on statistics that start off a 16-byte boundary."""
import numpy as np
import pytest

from oracle import densify as OD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(3, 9), (255, 9), (256, 16), (257, 1), (1025, 16), (4099, 4)])
def test_select_and_apply(n, k):
    import torch
    from paper_2410_20686_gb300.densify import DensifyParams, DensifyStats, apply, select
    rng = np.random.default_rng(n)
    count = rng.integers(0, 4, n).astype(np.int32)
    elev = (rng.uniform(0, 1, n) * count).astype(np.float32)
    grad = (rng.uniform(0, 2e-4, n) * count).astype(np.float32)
    means, scales = rng.normal(size=(n, 3)).astype(np.float32), rng.uniform(1e-4, 3e-3, (n, 3)).astype(np.float32)
    quats, opac = rng.normal(size=(n, 4)).astype(np.float32), rng.uniform(0.0, 0.05, n).astype(np.float32)
    sh, noise = rng.normal(size=(n, k, 3)).astype(np.float32), rng.normal(size=(n, 2, 3)).astype(np.float32)
    prm = DensifyParams(scene_extent=1.5)
    ref = OD.select(grad, elev, count, scales, opac, OD.DensifyParams(**prm.__dict__))
    for off in (0, 1):  # one element past an aligned start: the 4-byte loads
        st = DensifyStats(n + 1)
        for name, a in (("grad", grad), ("elev", elev), ("count", count)):
            t = getattr(st, name)[off:off + n]
            setattr(st, name, t.copy_(torch.from_numpy(a)))
        act = select(st, torch.from_numpy(scales).cuda(), torch.from_numpy(opac).cuda(), prm)
        np.testing.assert_array_equal(act.cpu().numpy(), ref)
    out = apply(*[torch.from_numpy(a).cuda() for a in (means, scales, quats, opac, sh)], act,
                torch.from_numpy(noise).cuda())
    want = OD.apply(means, scales, quats, opac, sh, ref, noise)
    plain = int(((ref == 0) | (ref == 1)).sum() + (ref == 1).sum())
    for i, (a, b) in enumerate(zip(out, want)):
        a = a.cpu().numpy()
        assert a.shape == b.shape
        if i < 2:  # children's means and scales: a few float32 roundings of values below about 10
            np.testing.assert_array_equal(a[:plain], b[:plain].astype(np.float32))
            np.testing.assert_allclose(a[plain:], b[plain:], rtol=1e-5, atol=1e-5)
        else:
            np.testing.assert_array_equal(a, b.astype(np.float32))
