"""A refresh walks a compacted list of samples with a bounded number of CTAs (forward.cu, slater.cu,
project.cu): more samples than CTAs, and samples that are not on the list, keep the bits of a load."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,B", [("hubbard4x4", 1500), ("hubbard8x8", 1300), ("tj8x8", 300)])
def test_refresh_keeps_the_bits_of_a_load(name, B):
    import torch
    pb = I.workload(name)
    ctx, _, occ, _ = setup(pb, B, 3, 4)
    bad = occ.copy()
    bad[::7] = 0  # no electrons: never on the list
    st = torch.empty(B, dtype=torch.int32, device="cuda")
    ctx.scale_load(torch.from_numpy(bad).cuda(), st)
    mv = torch.from_numpy(I.random_hop_moves(pb, occ, 3)[:, None, :].copy()).cuda()
    loaded = *ctx.log_psi(), ctx.ratios(mv), ctx.local_energy()
    ctx.scale_refresh(True)
    for a, b in zip(loaded, (*ctx.log_psi(), ctx.ratios(mv), ctx.local_energy())):
        assert torch.equal(torch.nan_to_num(a.double(), nan=3.0), torch.nan_to_num(b.double(), nan=3.0))
    assert torch.isfinite(loaded[3]).sum() > B // 2 and (st[::7] != 0).all()
