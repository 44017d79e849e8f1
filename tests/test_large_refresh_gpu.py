"""FP64 inverses above 1024 rows: a load takes one CTA per matrix (k_gj), a refresh a cluster of eight
(k_gj_cluster) up to the 1443 rows its panels leave room for. Both apply the same operations in the same
order, so the bits are equal, and a singular matrix among the others changes nothing for them."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,ne,prec", [(24, 1025, I.PREC_FP64), (24, 1040, I.PREC_MIXED), (28, 1460, I.PREC_FP64)])
def test_refresh_reproduces_load(L, ne, prec):
    import torch
    from paper_2604_25775_gb300 import binding as Bd
    pb = I.Problem(L, L, 1, 1, (ne + 1) // 2, ne // 2, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 1, 1, [1], [0], I.ACT_TANH, 1,
                   prec, 64, 1e-10)
    rng = np.random.default_rng(ne)
    M0 = rng.normal(size=(2 * pb.N, ne)) / np.sqrt(ne)
    occ = I.random_configs(pb, 3, 1)
    only = [i for i in range(pb.N) if occ[1, i] & 1 and not (occ[0, i] & 1 or occ[2, i] & 1)]
    if ne == 1040:
        M0[only[0]] = 0.0  # an orbital of the second walker alone
    ref = np.array([np.linalg.slogdet(M0[[s * pb.N + i for s in range(2) for i in range(pb.N) if (x[i] >> s) & 1]])[1]
                    for x in occ])
    mv = torch.from_numpy(I.random_hop_moves(pb, occ, 3)[:, None, :].copy()).cuda()
    ctx = Bd.make_context(pb, np.zeros(I.param_count(pb)), M0, 3)
    st = torch.empty(3, dtype=torch.int32, device="cuda")
    ctx.scale_load(torch.from_numpy(occ).cuda(), st)
    loaded = *ctx.log_psi(), ctx.ratios(mv)
    ctx.scale_refresh(True)
    refreshed = *ctx.log_psi(), ctx.ratios(mv)
    assert st.tolist() == ([0, 4, 0] if ne == 1040 else [0, 0, 0])
    live = st.cpu().numpy() == 0
    assert np.abs(loaded[0].cpu().numpy()[live] - ref[live]).max() <= (1e-8 if prec == I.PREC_FP64 else 1e-2)
    for a, b in zip(loaded, refreshed):
        assert torch.equal(torch.nan_to_num(a.double()), torch.nan_to_num(b.double()))
