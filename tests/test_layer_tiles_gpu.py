"""FP32 forward layers (forward.cu): one output per thread for few samples, 4 x 4 register tiles for many, in
the same order of summation, so a walker's log|psi| and local energy have the same bits either way: sites
off the tile of four, widths off 16, open edges, the stencils and a second convolution."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,h,pbc,ks,stencil,many", [(7, 7, 8, 1, [3, 1], 0, 430), (7, 5, 12, 0, [3, 3], 0, 400),
                                                         (9, 7, 16, 1, [3, 1], 0, 170), (7, 6, 20, 1, [5, 1], 1, 200),
                                                         (8, 8, 32, 1, [3, 3, 1], 0, 90), (5, 9, 64, 0, [3, 1], 0, 60)])
def test_few_and_many_samples_give_the_same_bits(Lx, Ly, h, pbc, ks, stencil, many):
    import torch
    n = Lx * Ly // 3
    assert 3 * Lx * Ly * h < 160 * 1024 < many * Lx * Ly * h and (Lx * Ly + 3) // 4 * (h // 4) >= 16
    pb = I.Problem(Lx, Ly, pbc, pbc, n, n - 1, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, len(ks), h, ks, [1] * len(ks),
                   I.ACT_TANH, 1, I.PREC_MIXED, 64, 1e-4, I.FAMILY_SCALE, 0, 0, 1e-5, stencil)
    occ = I.random_configs(pb, many, 11)
    ctx, _, _, _ = setup(pb, many, 5, 0, scale=0.1, occ=occ)
    few, _, _, _ = setup(pb, 3, 5, 0, scale=0.1, occ=occ[-3:].copy())
    (la, sg), (la3, sg3) = ctx.log_psi(), few.log_psi()
    assert torch.isfinite(la3).all()
    assert torch.equal(la[-3:], la3) and torch.equal(sg[-3:], sg3)
    if ks.count(3) < 2:
        assert torch.equal(ctx.local_energy()[-3:], few.local_energy())
