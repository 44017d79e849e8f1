"""The tiled forward layer and Slater-matrix kernels (forward.cu, slater.cu) at the edges of their
tiles: channel counts off 4 and 16, odd electron numbers, row groups that straddle the spins, and
the stencils, against the oracle."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import binding as Bd
from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import conditioning, eloc_term_scale, rel_err, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [I.PREC_FP64, I.PREC_MIXED])
@pytest.mark.parametrize("h,up,dn,stencil,k0", [(1, 5, 5, 0, 3), (3, 7, 6, 0, 3), (4, 9, 2, 0, 3), (12, 13, 10, 0, 3),
                                                (15, 1, 0, 0, 1), (16, 16, 17, 0, 3), (17, 11, 12, 1, 5), (20, 4, 4, 0, 3),
                                                (32, 15, 15, 1, 5), (33, 6, 9, 0, 3), (49, 10, 10, 0, 3), (64, 18, 15, 0, 3)])
def test_layers_and_slater_matrices(prec, h, up, dn, stencil, k0):
    """log|psi| of the load (mode's projection) and E_loc of the full-recompute path (FP64
    projection) within cond x 8 x 2^-24 (mixed) or cond x 1e3 x 2^-53 (FP64), as in the parity tests."""
    ks, rs = I.scale_layout(2, ksize_first=k0)
    pb = I.Problem(6, 6, 1, 1, up, dn, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 2, h, ks, rs, I.ACT_TANH, 1, prec, 64, 1e-4,
                   I.FAMILY_SCALE, 0, 0, 1e-5, stencil)
    ctx, ora, occ, st = setup(pb, 7, 40 + h, 50 + h, scale=0.1)
    la, sg = ctx.log_psi()
    la_o, sg_o = ora.log_psi(occ)
    cond = conditioning(ora, occ)
    unit = 1e3 * 2.0 ** -53 if prec == I.PREC_FP64 else 8 * 2.0 ** -24
    good = cond * unit < 1e-2
    assert good.any()
    tol = cond * unit
    assert (sg.cpu().numpy()[good] == sg_o[good]).all()
    assert (np.abs(la.cpu().numpy() - la_o)[good] <= tol[good]).all()
    e = ctx.local_energy(Bd.PATH_FULL).cpu().numpy()
    e_o, _ = ora.local_energy(occ)
    scale = np.maximum(eloc_term_scale(ora, occ), 1.0)
    assert (np.abs(e - e_o)[good] <= (4 * tol * scale)[good]).all()
