"""One walker's moves on one CTA and shared by the CTAs of a cluster (eloc.cuh): the local energies
have the same bits whatever the number of walkers of a call."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,prec", [("hubbard4x4", None), ("hubbard8x8", None), ("tj8x8", I.PREC_FP64),
                                       ("hubbard8x8", I.PREC_MIXED_BF16), ("scale_plus16x16", None), ("tj32x32", None)])
def test_local_energies_do_not_depend_on_the_split(name, prec):
    import torch
    pb = I.workload(name)
    if prec is not None:
        pb = pb.replace(precision=prec)
    many = 160 if pb.N <= 64 else 40 if pb.N <= 256 else 3
    counts = [n for n in (160, 100, 40, 20, 3, 1) if n <= many]
    ctx, _, occ, _ = setup(pb, many, 3, 4)
    ref = ctx.local_energy().cpu().numpy()
    assert np.isfinite(ref).sum() >= many - 1
    for n in counts[1:]:
        ctx.scale_load(torch.from_numpy(np.ascontiguousarray(occ[:n])).cuda())
        assert np.array_equal(ctx.local_energy().cpu().numpy(), ref[:n], equal_nan=True)
