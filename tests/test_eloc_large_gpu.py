"""Low-rank local energies on the large lattices where a launch shape's move scratch and lists only just fit
shared memory (eloc.cuh), against the full-recompute path in FP64 (both within 1e-10 of the terms' scale)."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import binding as Bd
from paper_2604_25775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# 20 warps end between 2356 and 2367 sites (16 channels), 12 at 2460 (64) and, with the plus, at 3783 (32)
@pytest.mark.parametrize("Lx,Ly,h,stencil,k0", [(59, 40, 16, 0, 3), (62, 38, 16, 0, 3), (91, 26, 16, 0, 3), (82, 30, 64, 0, 3),
                                                (88, 43, 32, 1, 5), (64, 64, 16, 0, 3), (64, 64, 64, 1, 5)])
def test_shared_memory_edges(Lx, Ly, h, stencil, k0):
    import torch
    pb = I.Problem(Lx, Ly, 1, 1, 3, 3, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 2, h, [k0, 1], [1, 1], I.ACT_TANH, 1, I.PREC_FP64,
                   64, 1e-10, I.FAMILY_SCALE, 0, 0, 1e-5, stencil)
    rng = np.random.default_rng(h)
    M0 = rng.normal(size=(2 * pb.N, 6))
    occ = I.random_configs(pb, 2, 4)
    ctx = Bd.make_context(pb, I.random_params(pb, 3, 0.05), M0, 2)
    ctx.scale_load(torch.from_numpy(occ).cuda())
    low, full = ctx.local_energy(), ctx.local_energy(Bd.PATH_FULL)
    cond = max(np.linalg.cond(M0[[s * pb.N + i for s in range(2) for i in range(pb.N) if (x[i] >> s) & 1]]) for x in occ)
    assert cond < 1e3
    assert ((low - full).abs() <= 1e-10 * (1 + full.abs() + 24 * cond)).all()
