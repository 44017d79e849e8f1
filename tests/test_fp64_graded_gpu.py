"""FP64 determinants and inverses of matrices whose entries span many orders of magnitude within a row and
a column, where a product on the leading digits alone loses what FP64 arithmetic keeps: localised
orbitals, columns with a scale of their own per row, entries of wild size. Against extended precision
(numpy's long double), with the error of FP64 elimination on the same matrices as the bound.

The network's weights are zero, so Phi is the chosen reference orbitals' rows. Compared are the
medians and the 90% quantiles over the walkers, which FP64 elimination in another order (LAPACK's
blocks, multiply-adds rounded once or twice) moves by less than 4x and 8x at these counts."""
import numpy as np
import pytest

from paper_2604_25775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(ne, prec=I.PREC_FP64):
    L = 8 if ne <= 64 else 16
    return I.Problem(L, L, 1, 1, (ne + 1) // 2, ne // 2, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 1, 1, [1], [0], I.ACT_TANH,
                     1, prec, 64, 1e-10)


def _orbitals(kind, pb, rng):
    N, n = pb.N, pb.Ne
    M = rng.normal(size=(2 * N, n))
    if kind[0] == "decay":  # exp(-d / xi) in the distance to a centre of the orbital's own, both spins alike
        c = rng.permutation(N)[np.arange(n) % N]
        i = np.arange(2 * N) % N
        d = [np.abs(a[:, None] - b[None, :]) for a, b in ((i % pb.Lx, c % pb.Lx), (i // pb.Lx, c // pb.Lx))]
        d = np.hypot(*(np.minimum(x, pb.Lx - x) for x in d))
        M = np.exp(-d / kind[1]) * (1 + 0.1 * M)
    elif kind[0] == "columns":  # some columns times a power of two of each row's own
        for q in range(kind[1]):
            M[:, 5 * q % n] *= np.exp2(rng.integers(0, kind[2] + 1, size=2 * N))
    else:
        M *= np.exp(kind[1] * rng.normal(size=M.shape))
    return M


def _orbs(x, N):
    return [s * N + i for s in range(2) for i in range(N) if (x[i] >> s) & 1]


def _eliminate(A, a, T):
    """log|det A|, its sign and the a-th column of its inverse by Gauss-Jordan with partial pivoting in type T."""
    n = len(A)
    M = np.concatenate([A, np.eye(n)[:, a:a + 1]], 1).astype(T)
    la, sg = T(0), 1
    for k in range(n):
        p = k + int(np.argmax(np.abs(M[k:, k])))
        if p != k:
            M[[k, p]] = M[[p, k]]
            sg = -sg
        la += np.log(np.abs(M[k, k]))
        sg = -sg if M[k, k] < 0 else sg
        f = M[:, k] / M[k, k]
        f[k] = 0
        M[:, k:] -= f[:, None] * M[k, k:]
    return la, sg, M[:, n] / np.diag(M)


KINDS = [("decay", 0.5), ("decay", 0.3), ("columns", 1, 20), ("columns", 1, 40), ("columns", 1, 90), ("columns", 8, 40),
         ("entries", 5.0)]


@pytest.mark.parametrize("kind", KINDS, ids=str)
@pytest.mark.parametrize("ne,B", [(56, 64), (33, 48), (160, 20)])
def test_graded_matrices(ne, B, kind):
    import torch
    from paper_2604_25775_gb300 import binding as Bd
    pb = _problem(ne)
    rng = np.random.default_rng(17 * ne + KINDS.index(kind))
    M0 = _orbitals(kind, pb, rng)
    occ = I.random_configs(pb, B, 3)
    mv = I.random_hop_moves(pb, occ, 5)
    ctx = Bd.make_context(pb, np.zeros(I.param_count(pb)), M0, B)
    st = torch.empty(B, dtype=torch.int32, device="cuda")
    ctx.scale_load(torch.from_numpy(occ).cuda(), st)
    la, sg = (x.cpu().numpy() for x in ctx.log_psi())
    r = ctx.ratios(torch.from_numpy(mv[:, None, :].copy()).cuda()).cpu().numpy()[:, 0]
    det = ctx.log_psi_sym(torch.arange(2 * pb.N, dtype=torch.int32, device="cuda")[None], torch.ones(1, dtype=torch.float64, device="cuda"))
    assert (st.cpu().numpy() == 0).all()
    err, bound = {"log": [], "det": [], "ratio": []}, {"log": [], "ratio": []}
    for b in range(B):
        Phi = M0[_orbs(occ[b], pb.N)]
        _, src, dst, s = mv[b]
        a = _orbs(occ[b], pb.N).index(s * pb.N + src)
        after = I.apply_moves(occ[b:b + 1], mv[b:b + 1])[0]
        sgn = (-1) ** sum(min(src, dst) < o - s * pb.N < max(src, dst) for o in _orbs(occ[b], pb.N) if s * pb.N <= o < (s + 1) * pb.N)
        assert (after != occ[b]).sum() == 2
        exact, plain = ((la_, sg_, np.sum(M0[s * pb.N + dst].astype(T) * y)) for T in (np.longdouble, np.float64)
                        for la_, sg_, y in [_eliminate(Phi, a, T)])
        assert sg[b] == exact[1] and int(det[1][b]) == exact[1]
        err["log"].append(abs(float(np.longdouble(la[b]) - exact[0])))
        err["det"].append(abs(float(np.longdouble(float(det[0][b])) - exact[0])))
        bound["log"].append(abs(float(np.longdouble(plain[0]) - exact[0])))
        scale = max(1.0, abs(float(exact[2])))
        err["ratio"].append(abs(float(np.longdouble(sgn * r[b]) - exact[2])) / scale)
        bound["ratio"].append(abs(float(np.longdouble(plain[2]) - exact[2])) / scale)
    bound["det"] = bound["log"]
    # what summing the logarithms of the pivots, or a row times a column, leaves in any order
    floor = {"log": 2.0 ** -50 * max(1.0, np.abs(la).max()), "ratio": 2.0 ** -53 * ne}
    floor["det"] = floor["log"]
    for k in err:
        for q, times in ((0.5, 4.0), (0.9, 8.0)):
            e, f = np.quantile(err[k], q), np.quantile(bound[k], q)
            print(f"{ne} {kind} {k} {q}: {e:.2e} (FP64 {f:.2e}, floor {floor[k]:.2e})")
            assert e <= times * f + floor[k], (k, q, e, f)


@pytest.mark.parametrize("kind", [("decay", 0.4), ("columns", 3, 60), ("rows", 150)], ids=str)
@pytest.mark.parametrize("ne,few,many", [(140, 9, 160), (200, 40, 160), (300, 9, 70), (530, 5, 70), (530, 20, 70)])
def test_graded_matrices_bit_for_bit_in_every_launch_shape(ne, few, many, kind):
    """What FP64 arithmetic takes of a product depends on the matrix alone, not on how clusters share it."""
    import torch
    from paper_2604_25775_gb300 import binding as Bd
    pb = _problem(ne) if ne <= 512 else _problem(ne).replace(Lx=24, Ly=24)
    rng = np.random.default_rng(ne)
    if kind[0] == "rows":
        M0 = rng.normal(size=(2 * pb.N, ne)) * np.exp2(rng.integers(-kind[1], kind[1] + 1, size=(2 * pb.N, 1)))
    else:
        M0 = _orbitals(kind, pb, rng)
    occ = I.random_configs(pb, many, 4)
    mv = torch.from_numpy(I.random_hop_moves(pb, occ, 8)[:, None, :].copy()).cuda()
    occ = torch.from_numpy(occ).cuda()
    out = []
    for B in (few, many):
        ctx = Bd.make_context(pb, np.zeros(I.param_count(pb)), M0, B)
        ctx.scale_load(occ[:B].contiguous(), torch.empty(B, dtype=torch.int32, device="cuda"))
        out.append((*ctx.log_psi(), ctx.ratios(mv[:B].contiguous())))
    for a, b in zip(*out):
        assert torch.equal(torch.nan_to_num(a.double()), torch.nan_to_num(b[:few].double()))


@pytest.mark.parametrize("h,spread", [(16, 40), (20, 90), (64, 40), (7, 20)])
def test_projection_of_channels_of_different_size(h, spread):
    """Phi = M0 + H W with H's channels times 2^0..2^spread and W's rows times the inverse: sums of terms of one
    size whose factors differ by `spread` bits. The layer hands the embedding rows on (no kernel, no
    bias, a residual), so H is the input."""
    import torch
    from paper_2604_25775_gb300 import binding as Bd
    ne, B = 24, 48
    pb = I.Problem(6, 6, 1, 1, 12, 12, I.MODEL_HUBBARD, 1.0, 0.0, 4.0, 0.0, 1, h, [1], [1], I.ACT_TANH, 1, I.PREC_FP64, 64,
                   1e-10)
    rng = np.random.default_rng(h)
    size = np.ldexp(1.0, rng.integers(0, spread + 1, size=h))
    params = np.zeros(I.param_count(pb))
    p = {k: params[o:o + int(np.prod(s))].reshape(s) for k, (o, s) in I.param_offsets(pb).items()}
    p["embed"][:] = rng.normal(size=(pb.N, 4, h)) * size
    p["proj_w"][:] = rng.normal(size=(h, 2 * ne)) / size[:, None]
    M0 = rng.normal(size=(2 * pb.N, ne))
    occ = I.random_configs(pb, B, 2)
    ctx = Bd.make_context(pb, params, M0, B)
    st = torch.empty(B, dtype=torch.int32, device="cuda")
    ctx.scale_load(torch.from_numpy(occ).cuda(), st)
    la, sg = (x.cpu().numpy() for x in ctx.log_psi())
    assert (st.cpu().numpy() == 0).all()
    err, bound = [], []
    for b in range(B):
        res = []
        for T in (np.longdouble, np.float64):
            H = p["embed"][np.arange(pb.N), occ[b]].astype(T)
            rows = []
            for o in _orbs(occ[b], pb.N):
                s, i = divmod(o, pb.N)
                x = M0[o].astype(T)
                for c in range(h):
                    x = x + H[i, c] * p["proj_w"][c, s * ne:(s + 1) * ne].astype(T)
                rows.append(x)
            res.append(_eliminate(np.stack(rows), 0, T))
        assert sg[b] == res[0][1]
        err.append(abs(float(np.longdouble(la[b]) - res[0][0])))
        bound.append(abs(float(np.longdouble(res[1][0]) - res[0][0])))
    floor = 2.0 ** -50 * max(1.0, np.abs(la).max())
    for q, times in ((0.5, 4.0), (0.9, 8.0)):
        print(f"h {h}: {np.quantile(err, q):.2e} (FP64 {np.quantile(bound, q):.2e}, floor {floor:.2e})")
        assert np.quantile(err, q) <= times * np.quantile(bound, q) + floor
