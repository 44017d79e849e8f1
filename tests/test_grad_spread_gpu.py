"""FP64 gradients of few walkers whose layers have more register tiles than a CTA's threads are spread over
several CTAs, those of many take one CTA each (grad.cu): the same sums in the same order but for the
bias, so few and many agree within rounding (N sums of terms up to the largest entry: N x 2^-50 of it)."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,h,pbc", [(11, 6, 32, 1), (13, 5, 32, 0), (16, 8, 24, 1), (9, 7, 40, 0), (8, 8, 32, 1)])
@pytest.mark.parametrize("recompute", [False, True])
def test_few_and_many_walkers_agree(Lx, Ly, h, pbc, recompute):
    import torch
    n = Lx * Ly // 4
    pb = I.Problem(Lx, Ly, pbc, pbc, n, n - 1, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 3, h, [3, 3, 1], [0, 1, 1], I.ACT_TANH,
                   1, I.PREC_FP64, 64, 1e-10)
    occ = I.random_configs(pb, 77, 6)
    many, _, _, st = setup(pb, 77, 5, 0, scale=0.1, occ=occ)
    few, _, _, _ = setup(pb, 76, 5, 0, scale=0.1, occ=occ[:76].copy())
    a, b = many.grad_logpsi(recompute)[:76], few.grad_logpsi(recompute)
    live = torch.from_numpy(st[:76] == 0).cuda()
    assert live.any()
    scale = b.abs().amax(1, keepdim=True)
    assert ((a - b).abs() <= Lx * Ly * 2.0 ** -50 * scale)[live].all()
