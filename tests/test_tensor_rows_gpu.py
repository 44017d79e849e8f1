"""Rows of the tensor-core layers (ace.cu): gathered from split rows or read as blocked tiles, with row
counts off the 128 of a tile, open edges and lattices narrower than the stencil, against the oracle."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import binding as Bd
from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import conditioning, eloc_term_scale, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,Lx,Ly,px,py,up,dn,B", [("scale_l16x16", 5, 3, 1, 0, 4, 3, 1), ("scale_l16x16", 5, 5, 1, 1, 2, 2, 9),
                                                      ("scale_l16x16", 7, 3, 0, 0, 3, 5, 6), ("ace8x8", 5, 3, 0, 1, 4, 3, 7),
                                                      ("ace16x16", 4, 2, 1, 0, 2, 3, 33), ("ace16x16", 16, 3, 1, 1, 4, 4, 8)])
def test_row_tiles(name, Lx, Ly, px, py, up, dn, B):
    """log|psi| within cond x 8 x 2^-24 per layer of the network (at most 18) and E_loc within 1e-4 of its term
    scale for cond(Phi) < 1e3, as in the parity tests."""
    pb = I.workload(name).replace(Lx=Lx, Ly=Ly, pbc_x=px, pbc_y=py, n_up=up, n_dn=dn)
    ctx, ora, occ, st = setup(pb, B, 80 + Lx, 90 + B, scale=0.02)
    cond = conditioning(ora, occ)
    good = (st == 0) & (cond < 1e3)
    assert good.any()
    la, sg = ctx.log_psi()
    la_o, sg_o = ora.log_psi(occ)
    assert (sg.cpu().numpy()[good] == sg_o[good]).all()
    assert (np.abs(la.cpu().numpy() - la_o)[good] <= (cond * 8 * 18 * 2.0 ** -24)[good]).all()
    e_o, _ = ora.local_energy(occ)
    scale = np.maximum(eloc_term_scale(ora, occ), 1.0)
    for path in [Bd.PATH_FULL] + ([Bd.PATH_LOWRANK] if name.startswith("scale") else []):
        e = ctx.local_energy(path).cpu().numpy()
        assert (np.abs(e - e_o)[good] <= 1e-4 * scale[good]).all()
