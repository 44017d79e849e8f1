"""The FP32 projector and G0t (project.cu) at electron numbers and widths on both sides of each register
tile: an output is one chain of multiply-adds whatever the tile, so a walker gives the same bits among many
walkers (the tile of the least padded area) as among few (the small tile), and its ratios agree with the
FP64 mode's within FP32's rounding of the inverse, cond x 64 x 2^-24."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import conditioning, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,h,ne,many", [(8, 32, 57, 60), (8, 32, 64, 60), (8, 17, 65, 60), (8, 3, 113, 60), (16, 32, 60, 24),
                                         (16, 32, 113, 24), (16, 64, 128, 24), (16, 16, 129, 24), (16, 33, 180, 24),
                                         (16, 32, 225, 24), (16, 32, 256, 24), (16, 5, 257, 24)])
def test_same_bits_in_every_tile(L, h, ne, many):
    import torch
    ks, rs = I.scale_layout(2)
    pb = I.Problem(L, L, 1, 1, (ne + 1) // 2, ne // 2, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 2, h, ks, rs, I.ACT_TANH, 1,
                   I.PREC_MIXED, 64, 1e-4)
    occ = I.random_configs(pb, many, ne)
    mv = I.random_hop_moves(pb, occ, 5)
    mv_d = torch.from_numpy(mv[:, None, :].copy()).cuda()
    ctx, ora, _, st = setup(pb, many, 7, 0, occ=occ)
    few, _, _, _ = setup(pb, 2, 7, 0, occ=occ[:2].copy())
    ref, _, _, _ = setup(pb.replace(precision=I.PREC_FP64), 2, 7, 0, occ=occ[:2].copy())
    assert (st == 0).all()
    r, r2, rr = ctx.ratios(mv_d), few.ratios(mv_d[:2].contiguous()), ref.ratios(mv_d[:2].contiguous())
    assert torch.equal(r[:2], r2)
    assert torch.equal(ctx.local_energy()[:2], few.local_energy())
    tol = torch.from_numpy(conditioning(ora, occ[:2]) * 64 * 2.0 ** -24).cuda()[:, None]
    good = tol < 1e-1
    assert good.any()
    assert ((r2 - rr).abs() <= tol * torch.clamp(rr.abs(), min=1.0))[good].all()
