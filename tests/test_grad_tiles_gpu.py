"""The staged gradient kernels (grad.cu) at the edges of their tiles -- odd site counts, the largest
staged lattice and the first beyond it, widths off 32, wide stencils, open edges -- against the
oracle's backward pass."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I
from tests.gpu_common import conditioning, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [I.PREC_FP64, I.PREC_MIXED])
@pytest.mark.parametrize("Lx,Ly,px,py,h,stencil,k", [(3, 3, 1, 1, 8, 0, 3), (5, 3, 1, 0, 24, 0, 3), (7, 9, 0, 0, 40, 0, 5),
                                                     (16, 8, 1, 1, 16, 1, 5), (11, 11, 1, 1, 64, 0, 3),
                                                     (12, 11, 1, 0, 8, 0, 3), (4, 4, 1, 1, 32, 0, 1)])
def test_staged_gradients(prec, Lx, Ly, px, py, h, stencil, k):
    """Relative to the sample's largest entry: FP64 within 1e-10 (cond(Phi) < 1e6), mixed 1e-4 (cond < 1e3),
    as in the parity tests; every entry written."""
    import torch
    N = Lx * Ly
    pb = I.Problem(Lx, Ly, px, py, (N + 3) // 4, N // 4, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 3, h, [k, k, 1], [1, 0, 1],
                   I.ACT_TANH, 1, prec, 64, 1e-4, I.FAMILY_SCALE, 0, 0, 1e-5, stencil)
    ctx, ora, occ, st = setup(pb, 9, 60 + h, 70 + h, scale=0.1)
    cond = conditioning(ora, occ)
    good = (st == 0) & (cond < (1e6 if prec == I.PREC_FP64 else 1e3))
    assert good.any()
    g_o = ora.grad_logpsi(occ)[good]
    scale = np.maximum(np.abs(g_o).max(axis=1, keepdims=True), 1.0)
    for recompute in (False, True):
        g_d = torch.full((ctx.B, ctx.P), float("nan"), dtype=torch.float64, device="cuda")
        ctx.scale_grad_logpsi(g_d, recompute)
        err = np.abs(g_d.cpu().numpy()[good] - g_o) / scale
        assert err.max() <= (1e-10 if prec == I.PREC_FP64 else 1e-4)
