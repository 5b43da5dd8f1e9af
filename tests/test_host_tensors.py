"""The device entry points refuse tensors that are not on a GPU, before anything is launched on their pointers."""
import pytest
import torch

from paper_2410_20686_gb300 import _lib as L
from paper_2410_20686_gb300 import densify as D
from paper_2410_20686_gb300.loss import l1_dssim


def _loss(lam):
    return lambda: l1_dssim([torch.rand(3, 8, 16)], [torch.rand(3, 8, 16)], lam=lam)


def _select():
    stats = D.DensifyStats(4, torch.device("cpu"))
    return D.select(stats, torch.rand(4, 3), torch.rand(4))


def _apply():
    return D.apply(torch.rand(4, 3), torch.rand(4, 3), torch.rand(4, 4), torch.rand(4), torch.rand(4, 1, 3),
                   torch.zeros(4, dtype=torch.uint8))


def _indexed():
    x = torch.rand(3, 8, 16, device="cpu:0")
    return l1_dssim([x], [x])


@pytest.mark.parametrize("call", [lambda: L.raw_stream(torch.device("cpu")), _loss(0.2), _loss(0.0), _select, _apply, _indexed],
                         ids=["stream", "loss", "l1", "select", "apply", "indexed"])
def test_host_tensors_are_refused(call):
    with pytest.raises(ValueError):
        call()
