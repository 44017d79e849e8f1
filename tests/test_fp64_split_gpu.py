"""FP64 elimination with its block products as split FP16 tensor-core products (dense_inverse.cu,
fp64_mma.cuh): log|det|, sign and inverse at the edges of its blocks (16 pivots), tiles (8
columns, 16 rows), launch shapes (128 / 256 / 512 / 1024 rows, clusters of 4 and 8 CTAs) and
scale rules, against numpy in FP64.

The network's weights are zero, so Phi is the chosen reference orbitals' rows; the tolerance is
the one of the other FP64 tests, cond(Phi) x 1e3 x 2^-53."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(ne, prec=I.PREC_FP64):
    L = 4 if ne <= 32 else 8 if ne <= 128 else 16 if ne <= 512 else 24
    up = (ne + 1) // 2
    return I.Problem(L, L, 1, 1, up, ne - up, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 1, 1, [1], [0], I.ACT_TANH, 1, prec,
                     64, 1e-10)


def _slater(M0, occ, N):
    return np.stack([M0[[s * N + i for s in range(2) for i in range(N) if (x[i] >> s) & 1]] for x in occ])


def _run(pb, M0, occ):
    import torch
    from paper_2604_25775_gb300 import binding as Bd
    ctx = Bd.make_context(pb, np.zeros(I.param_count(pb)), M0, len(occ))
    st = torch.empty(len(occ), dtype=torch.int32, device="cuda")
    ctx.scale_load(torch.from_numpy(occ).cuda(), st)
    la, sg = ctx.log_psi()
    return ctx, la.cpu().numpy(), sg.cpu().numpy(), st.cpu().numpy()


def _check_inverse(ctx, pb, M0, occ, Phi, tol):
    """Ratios of one hop per walker: one column of M0 Phi^-1."""
    import torch
    mv = I.random_hop_moves(pb, occ, 3)
    r = ctx.ratios(torch.from_numpy(mv[:, None, :].copy()).cuda()).cpu().numpy()[:, 0]
    after = I.apply_moves(occ, mv)
    det0, det1 = np.linalg.slogdet(Phi), np.linalg.slogdet(_slater(M0, after, pb.N))
    ref = det1[0] * det0[0] * np.exp(det1[1] - det0[1])
    live = mv[:, 0] >= 0
    assert (np.abs(r - ref)[live] <= (tol * np.maximum(1.0, np.abs(ref)))[live]).all()


@pytest.mark.parametrize("ne", [1, 2, 7, 8, 9, 15, 16, 17, 24, 31, 32, 33, 47, 49, 63, 64, 65, 127, 128, 129, 160, 223, 225,
                                255, 256, 257, 447, 449, 512, 513, 800, 1024, 1025])
def test_block_edges(ne):
    pb = _problem(ne)
    rng = np.random.default_rng(ne)
    M0 = rng.normal(size=(2 * pb.N, ne)) / np.sqrt(ne)
    B = 5 if ne > 128 else 12
    occ = I.random_configs(pb, B, 10 + ne)
    Phi = _slater(M0, occ, pb.N)
    tol = np.linalg.cond(Phi) * 1e3 * 2.0 ** -53
    ctx, la, sg, st = _run(pb, M0, occ)
    ref = np.linalg.slogdet(Phi)
    assert (st == 0).all()
    assert (sg == ref[0]).all()
    assert (np.abs(la - ref[1]) <= tol).all()
    if ne < 2 * pb.N:
        _check_inverse(ctx, pb, M0, occ, Phi, tol)
    if ne > 512:
        return
    # determinants alone (the full-recompute entry), many and few matrices a call
    e_low = ctx.local_energy(0).cpu().numpy()
    e_full = ctx.local_energy(1).cpu().numpy()
    n_terms = 8 * pb.N
    assert (np.abs(e_low - e_full) <= n_terms * tol * np.maximum(1.0, np.abs(e_full))).all()


@pytest.mark.parametrize("ne,spread", [(56, 60), (56, 140), (100, 140), (200, 90), (200, 150)])
def test_row_scales(ne, spread):
    """Rows of the reference orbitals multiplied by powers of two up to 2^+-spread: inside 2^+-100
    the split products take them, beyond it the plain FP64 block update. log|psi| moves by the
    exact sum of the exponents."""
    pb = _problem(ne)
    rng = np.random.default_rng(ne + spread)
    M0 = rng.normal(size=(2 * pb.N, ne)) / np.sqrt(ne)
    ex = rng.integers(-spread, spread + 1, size=2 * pb.N)
    occ = I.random_configs(pb, 6, 77)
    Phi = _slater(M0, occ, pb.N)
    tol = np.linalg.cond(Phi) * 1e3 * 2.0 ** -53
    ref = np.linalg.slogdet(Phi)
    shift = np.array([sum(ex[s * pb.N + i] for s in range(2) for i in range(pb.N) if (x[i] >> s) & 1) for x in occ])
    ctx, la, sg, st = _run(pb, np.ldexp(M0, ex[:, None]), occ)
    expect = ref[1] + shift * np.log(2.0)
    assert (st == 0).all() and (sg == ref[0]).all()
    assert (np.abs(la - expect) <= tol + 1e-13 * np.abs(expect)).all()


def test_zero_row_nan_and_infinity():
    """A zero row is singular; a NaN or an infinity reaches the result and no other walker."""
    ne = 40
    pb = _problem(ne)
    rng = np.random.default_rng(5)
    M0 = rng.normal(size=(2 * pb.N, ne))
    occ = I.random_configs(pb, 8, 9)
    hit = []
    for x in occ:  # an orbital only some walkers occupy
        hit.append(bool(x[3] & 1))
    assert any(hit) and not all(hit)
    ref = np.linalg.slogdet(_slater(M0, occ, pb.N))
    for bad in (0.0, np.nan, np.inf):
        M = M0.copy()
        M[3, :] = bad if bad == 0.0 else M[3, :]
        if bad != 0.0:
            M[3, 5] = bad
        ctx, la, sg, st = _run(pb, M, occ)
        for b, h in enumerate(hit):
            if not h:
                assert st[b] == 0 and sg[b] == ref[0][b] and abs(la[b] - ref[1][b]) <= 1e-9
            elif bad == 0.0:
                assert st[b] == 4 and sg[b] == 0 and np.isneginf(la[b])
            else:
                assert not np.isfinite(la[b])


@pytest.mark.parametrize("ne,many", [(140, 160), (140, 60), (300, 70), (460, 70), (530, 20), (530, 70)])
def test_launch_shapes_agree_bit_for_bit(ne, many):
    """A matrix gives the same bits alone (a cluster of CTAs) and among many (one CTA each)."""
    import torch
    pb = _problem(ne, I.PREC_MIXED)
    rng = np.random.default_rng(ne)
    M0 = rng.normal(size=(2 * pb.N, ne)) / np.sqrt(ne)
    occ = I.random_configs(pb, many, 4)
    mv = torch.from_numpy(I.random_hop_moves(pb, occ, 8)[:, None, :].copy()).cuda()
    ctx, la, sg, _ = _run(pb, M0, occ)
    r = ctx.ratios(mv).cpu().numpy()
    few, la2, sg2, _ = _run(pb, M0, occ[:3])
    r2 = few.ratios(mv[:3].contiguous()).cpu().numpy()
    assert np.array_equal(la[:3], la2) and np.array_equal(sg[:3], sg2) and np.array_equal(r[:3], r2)
