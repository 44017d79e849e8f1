"""FP64 inverses shared by a cluster of CTAs (dense_inverse.cu) while other work keeps their SMs busy:
the CTAs of a cluster run apart from one another, and every one still has to read a block's columns
before their owner stores them swept. The bits are those of the same matrices inverted by one CTA
each; a singular matrix among the others leaves them alone."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(ne):
    L = 16 if ne <= 512 else 24
    return I.Problem(L, L, 1, 1, ne // 2, ne - ne // 2, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 1, 1, [1], [0], I.ACT_TANH,
                     1, I.PREC_FP64, 64, 1e-10)


def _results(ctx, occ, mv):
    import torch
    st = torch.empty(len(occ), dtype=torch.int32, device="cuda")
    ctx.scale_load(occ, st)
    la, sg = ctx.log_psi()
    return la, sg, st, ctx.ratios(mv)


# clusters of 4 and 2 up to 256 rows, of 4 up to 512, of 8 and 4 above
@pytest.mark.parametrize("ne,few,many", [(130, 9, 160), (224, 30, 160), (225, 60, 160), (448, 20, 70), (530, 6, 70),
                                         (530, 30, 70)])
def test_cluster_inverse_beside_other_work(ne, few, many):
    import torch
    from paper_2604_25775_gb300 import binding as Bd
    pb = _problem(ne)
    rng = np.random.default_rng(ne + few)
    M0 = rng.normal(size=(2 * pb.N, ne)) / np.sqrt(ne)
    occ = I.random_configs(pb, many, 4)
    M0[pb.N + 5] = 0.0  # singular where the down spin of site 5 is there
    bad = (occ[:, 5] >> 1).astype(bool)
    assert bad[:few].any() and not bad[:few].all()
    mv = torch.from_numpy(I.random_hop_moves(pb, occ, 8)[:, None, :].copy()).cuda()
    occ = torch.from_numpy(occ).cuda()
    params = np.zeros(I.param_count(pb))
    ref = _results(Bd.make_context(pb, params, M0, many), occ, mv)
    assert ((ref[2].cpu().numpy() == 4) == bad).all()
    ctx = Bd.make_context(pb, params, M0, few)
    ours = torch.cuda.current_stream()
    other = torch.cuda.Stream()
    x = torch.randn(1 << 24, device="cuda")
    torch.cuda.synchronize()
    for _ in range(12):
        with torch.cuda.stream(other):
            for _ in range(20):
                x.sin_()
        got = _results(ctx, occ[:few].contiguous(), mv[:few].contiguous())
        for a, b in zip(got, ref):
            assert torch.equal(torch.nan_to_num(a, nan=7.0) if a.is_floating_point() else a,
                               torch.nan_to_num(b[:few], nan=7.0) if b.is_floating_point() else b[:few])
    ours.wait_stream(other)
    torch.cuda.synchronize()
