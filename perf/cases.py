"""The work that programs ask of this framework, as cases that can be timed and compared.

Every case is one call (or one short call sequence) of a variational Monte Carlo program on a
lattice-fermion system: local energies of resident walkers, a chain step's commits, a
Metropolis sweep, a load, per-sample gradients, the full-recompute comparison path, a
symmetry-projected amplitude, and the amplitudes of the ACE and local energies of the wide
SCALE networks. Systems and networks are the named workloads of `inputs.workload`.

Walkers are draws of the workload's reference determinant, |det(M0 rows)|^2 (up spins, then
down spins; t-J: the down spins on the sites the up spins left), which is what a program
starts its chains from; weights are the N(0, 0.05^2) draws of `inputs.random_params`
(N(0, 0.02^2) for the ACE and wide networks, as in bench.py, and for the deep stack of convolutions,
which keeps the state near that determinant).

The library returns float64 in every mode. In the mixed modes the network, the ratios and the
cached inverse are FP32, so a program keeps those results in float32, and so do the cases; the
FP64 mode's results stay float64.
"""
from __future__ import annotations

import math

import torch

from paper_2604_25775_gb300 import autograd as A
from paper_2604_25775_gb300 import binding as Bd
from paper_2604_25775_gb300 import inputs as I


def listed():
    return [
        # the smallest request of a served chain: 64 walkers on 8x8, latency counts
        {"name": "energy_8x8", "op": "energy", "system": "hubbard8x8", "walkers": 64},
        # the main path at a production batch: 16x16, 1/8 doping, FP16x3 site-wise layers
        {"name": "energy_16x16", "op": "energy", "system": "hubbard16x16", "walkers": 4096},
        # t-J on the largest served lattice, a ragged chain
        {"name": "energy_tj_32x32", "op": "energy", "system": "tj32x32", "walkers": 133},
        # SCALE-L widths: the cached update as row GEMMs
        {"name": "energy_scale_l", "op": "energy", "system": "scale_l16x16", "walkers": 24},
        # accepted moves of a chain step: a Woodbury commit per walker, there and back
        {"name": "commit_16x16", "op": "commit", "system": "hubbard16x16", "walkers": 2048},
        # sampling between energy evaluations
        {"name": "sweep_16x16", "op": "sweep", "system": "hubbard16x16", "walkers": 1024, "steps": 16},
        # new walkers, or a resumed run: forward, FP64 inverse, projector
        {"name": "load_16x16", "op": "load", "system": "hubbard16x16", "walkers": 1500},
        # local energies by full recompute: the comparison path
        {"name": "full_16x16", "op": "full", "system": "hubbard16x16", "walkers": 4},
        # per-sample gradients of the deep stack on the cylinder, mixed precision
        {"name": "grad_16x4", "op": "grad", "system": "cylinder16x4", "precision": "mixed", "walkers": 512,
         "recompute": False},
        # one variational update in FP64: new weights, load, per-sample gradients
        {"name": "update_fp64_8x8", "op": "update", "system": "hubbard8x8", "precision": "fp64", "walkers": 200,
         "recompute": False},
        # projection onto the translations by two sites
        {"name": "symmetry_16x16", "op": "symmetry", "system": "hubbard16x16", "walkers": 100, "stride": 2},
        # amplitudes of the ACE network at its published widths
        {"name": "ace_16x16", "op": "load", "system": "ace16x16", "walkers": 96},
    ]


PRECISIONS = {"fp64": I.PREC_FP64, "mixed": I.PREC_MIXED, "mixed_fp16": I.PREC_MIXED_FP16,
              "mixed_bf16": I.PREC_MIXED_BF16}


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["energy"] * 4 + ["commit", "sweep", "load", "load", "full", "grad", "update", "symmetry"])
    if op == "energy":
        system, most = rng.choice([("hubbard4x4", 8192), ("hubbard8x8", 8192), ("tj8x8", 8192), ("hubbard_ph8x8", 8192),
                                   ("hubbard16x16", 4096), ("tj16x16", 4096), ("scale_plus16x16", 2048),
                                   ("hubbard32x32", 120), ("tj32x32", 133), ("scale_l8x8", 96), ("scale_l16x16", 24)])
        case = {"op": op, "system": system, "walkers": _log(rng, 1, most)}
        if system in ("hubbard8x8", "tj8x8", "hubbard16x16"):
            case["precision"] = rng.choice(["mixed", "mixed_fp16", "mixed_bf16"])
        return case
    if op in ("commit", "sweep"):
        system, most = rng.choice([("hubbard8x8", 4096), ("hubbard8x8", 4096), ("hubbard16x16", 2048),
                                   ("hubbard32x32", 64)])
        case = {"op": op, "system": system, "walkers": _log(rng, 1, most)}
        if op == "sweep":
            case["steps"] = _log(rng, 1, 16)
            case["walkers"] = max(1, case["walkers"] // 2)
        return case
    if op == "load":
        system, most = rng.choice([("hubbard8x8", 8192), ("tj16x16", 1500), ("hubbard16x16", 1500),
                                   ("hubbard32x32", 48), ("ace8x8", 512), ("ace16x16", 96), ("scale_l16x16", 96)])
        return {"op": op, "system": system, "walkers": _log(rng, 1, most)}
    if op == "full":
        system, most = rng.choice([("hubbard4x4", 256), ("hubbard8x8", 96), ("tj8x8", 96), ("hubbard16x16", 4)])
        return {"op": op, "system": system, "walkers": _log(rng, 1, most)}
    if op in ("grad", "update"):
        system, most = rng.choice([("cylinder16x4", 512), ("hubbard8x8", 1024), ("hubbard16x16", 300)])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        if precision == "fp64":
            most //= 4
        return {"op": op, "system": system, "precision": precision, "walkers": _log(rng, 1, most),
                "recompute": bool(rng.random() < 0.3)}
    system, most = rng.choice([("hubbard8x8", 512), ("tj8x8", 512), ("hubbard16x16", 100)])
    return {"op": op, "system": system, "walkers": _log(rng, 1, most), "stride": 2 if system == "hubbard16x16" else 1}


def _problem(case):
    pb = I.workload(case["system"])
    if case.get("precision"):
        pb = pb.replace(precision=PRECISIONS[case["precision"]], drift_tol=1e-10 if case["precision"] == "fp64" else 1e-4)
    return pb


def _keep(pb, x):
    """The type a program keeps a result in: the precision the mode computes in."""
    return x if pb.precision == I.PREC_FP64 else x.float()


# ---- inputs, from the seed alone ---------------------------------------------------------
def _draw_sites(V, free, gen):
    """One site set per row from |det V[sites]|^2 (V [N][n] orthonormal columns): sites one by
    one with the probability of the chain rule, restricted to the `free` sites [B][N]."""
    B, (N, n) = free.shape[0], V.shape
    K = V @ V.T
    d = torch.diagonal(K).expand(B, N).clone()
    L = torch.zeros(B, N, n, dtype=torch.float64, device="cuda")
    occ = torch.zeros(B, N, dtype=torch.bool, device="cuda")
    u = torch.rand(n, B, 1, dtype=torch.float64, device="cuda", generator=gen)
    rows = torch.arange(B, device="cuda")
    for t in range(n):
        p = (d.clamp(min=0.0) * free * ~occ).cumsum(1)
        i = torch.searchsorted(p, u[t] * p[:, -1:]).clamp(max=N - 1)[:, 0]
        col = K[i] - torch.bmm(L[:, :, :t], L[rows, i, :t].unsqueeze(2)).squeeze(2)
        L[:, :, t] = col / d[rows, i].clamp(min=1e-12).sqrt().unsqueeze(1)
        d = d - L[:, :, t].square()
        occ[rows, i] = True
    return occ


def _inputs(case, seed):
    pb = _problem(case)
    deep = pb.family != I.FAMILY_SCALE or sum(int(k) > 1 for k in pb.ksize) > 1
    params = torch.from_numpy(I.random_params(pb, seed, 0.02 if deep else 0.05)).cuda()
    M0 = torch.from_numpy(I.plane_wave_M0(pb)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B, N = case["walkers"], pb.N
    of = 8 if case["op"] in ("grad", "update") else 1
    everywhere = torch.ones(B * of, N, dtype=torch.bool, device="cuda")
    up = _draw_sites(M0[:N, :pb.n_up], everywhere, gen)
    dn = _draw_sites(M0[N:, pb.n_up:], ~up if pb.model == I.MODEL_TJ else everywhere, gen)
    occ = up.to(torch.int8) + 2 * dn.to(torch.int8)
    if of > 1:
        # gradients weigh a walker with a small amplitude most, which a chain rarely visits: the
        # draw of the largest |psi| among eight
        logabs = _Model64(pb, params, M0).log_psi(occ)[0].view(B, of)
        occ = occ.view(B, of, N)[torch.arange(B, device="cuda"), logabs.argmax(1)]
    return pb, params, M0, occ.contiguous(), gen


def _bonds(pb):
    """[(i, j)] of the nearest-neighbour bonds, then of the next-nearest ones where t' != 0."""
    nn, nnn = [], []
    for bonds, steps in ((nn, ((1, 0), (0, 1))), (nnn, ((1, 1), (1, -1)) if pb.tp else ())):
        for i in range(pb.N):
            for dx, dy in steps:
                j = _site(pb, i, dx, dy)
                if j >= 0:
                    bonds.append((i, j))
    return nn, nnn


def _site(pb, i, dx, dy):
    x, y = i % pb.Lx + dx, i // pb.Lx + dy
    if not (0 <= x < pb.Lx or pb.pbc_x) or not (0 <= y < pb.Ly or pb.pbc_y):
        return -1
    return (y % pb.Ly) * pb.Lx + x % pb.Lx


def _accepted_moves(pb, M0, occ, gen):
    """A nearest-neighbour hop per walker with the weight min(1, ratio^2) of the reference
    determinant: the moves that a Metropolis step accepts."""
    nn = torch.tensor(_bonds(pb)[0], device="cuda")
    both = torch.cat([nn, nn.flip(1)])
    src, dst = both[:, 0], both[:, 1]
    weight = []
    for s, n, V in ((0, pb.n_up, M0[:pb.N, :pb.n_up]), (1, pb.n_dn, M0[pb.N:, pb.n_up:])):
        on = (occ >> s & 1).bool()
        sites = on.nonzero()[:, 1].view(-1, n)
        G = V @ torch.linalg.inv(V[sites])  # [B][site][electron]
        slot = on.cumsum(1) - 1
        ratio = G[torch.arange(len(occ), device="cuda")[:, None], dst[None, :], slot[:, src].clamp(min=0)]
        ok = on[:, src] & ~on[:, dst]
        if pb.model == I.MODEL_TJ:
            ok &= occ[:, dst] == 0
        weight.append(ratio.square().clamp(max=1.0) * ok)
    pick = torch.multinomial(torch.cat(weight, 1), 1, generator=gen)[:, 0]
    m, s = pick % len(both), pick // len(both)
    there = torch.stack([torch.zeros_like(m), src[m], dst[m], s], 1).int().contiguous()
    back = torch.stack([torch.zeros_like(m), dst[m], src[m], s], 1).int().contiguous()
    return there, back


def _group(pb, stride):
    """Translations by multiples of `stride` sites along both axes."""
    perms = I.symmetry_group(pb, translations=True)
    keep = [g for g, p in enumerate(perms) if p[0] % pb.Lx % stride == 0 and p[0] // pb.Lx % stride == 0]
    return torch.from_numpy(perms[keep]).cuda()


def prepare(case, seed):
    pb, params, M0, occ, gen = _inputs(case, seed)
    op, B = case["op"], case["walkers"]
    ctx = Bd.Context(pb, B)
    ctx.scale_set_params(params, M0)
    s = {"op": op, "pb": pb, "ctx": ctx, "params": params, "M0": M0, "occ": occ}
    if op == "load":
        s["status"] = torch.empty(B, dtype=torch.int32, device="cuda")
    elif op != "update":
        ctx.scale_load(occ)
    if op == "commit":
        s["moves"] = _accepted_moves(pb, M0, occ, gen)
    elif op == "sweep":
        s["random"] = [torch.from_numpy(x).cuda() for x in I.metropolis_randoms(pb, B, case["steps"], seed)]
    elif op == "symmetry":
        s["perms"] = _group(pb, case["stride"])
        s["chi"] = torch.ones(len(s["perms"]), dtype=torch.float64, device="cuda")
    elif op in ("grad", "update"):
        s["recompute"] = case["recompute"]
    return s


# ---- one pass through the public entry points ---------------------------------------------
def run(s):
    op, pb, ctx = s["op"], s["pb"], s["ctx"]
    if op == "energy":
        return _keep(pb, ctx.local_energy())
    if op == "full":
        return _keep(pb, ctx.local_energy(Bd.PATH_FULL))
    if op == "load":
        ctx.scale_load(s["occ"], s["status"])
        logabs, sign = ctx.log_psi()
        return _keep(pb, logabs), sign, s["status"]
    if op == "commit":
        there, back = s["moves"]
        ctx.scale_commit(there)
        la1, sg1 = ctx.log_psi()
        ctx.scale_commit(back)
        la2, sg2 = ctx.log_psi()
        return _keep(pb, la1), sg1, _keep(pb, la2), sg2, ctx.get_occ()
    if op == "sweep":
        accepted = ctx.sweep(*s["random"])
        logabs, sign = ctx.log_psi()
        return accepted, ctx.get_occ(), _keep(pb, logabs), sign
    if op == "symmetry":
        logabs, sign = ctx.log_psi_sym(s["perms"], s["chi"])
        return _keep(pb, logabs), sign
    if op == "grad":
        return _keep(pb, ctx.grad_logpsi(s["recompute"]))
    return _keep(pb, A.per_sample_gradients(s["params"], s["occ"], s["M0"], ctx, s["recompute"]))


# ---- what a pass cannot do without ----------------------------------------------------------
def work(case):
    pb = _problem(case)
    B, N, Ne, T = case["walkers"], pb.N, pb.Ne, 8 if pb.precision == I.PREC_FP64 else 4
    out = T  # bytes of one returned value (see _keep)
    wide = pb.family != I.FAMILY_SCALE
    h, hl = pb.h, I.layer_widths(pb, pb.n_layers - 1)[1]
    taps = [len(I.stencil_taps(int(k), pb.stencil)) for k in pb.ksize]
    layer = [2.0 * taps[l] * math.prod(I.layer_widths(pb, l)) for l in range(pb.n_layers)]  # flop of a site
    site_wise = sum(layer[1:])
    n_params = I.param_count(pb)
    # expected connected configurations and electrons on the affected sites of a move
    fu, fd = pb.n_up / N, pb.n_dn / N
    nn, nnn = (len(b) for b in _bonds(pb))
    if pb.model == I.MODEL_TJ:
        moves = nn * 2 * (fu + fd) * (1 - fu - fd) + nn * 2 * fu * fd
    else:
        moves = (nn + nnn) * 2 * (fu * (1 - fu) + fd * (1 - fd))
    S = {9: 12, 13: 18}.get(taps[0], 2)
    r = S * (fu + fd)
    cache = T * (Ne * Ne + 2 * N * h) + N + 8 * N
    forward = N * sum(layer) + 2.0 * Ne * Ne * hl
    lu, inverse = 2.0 / 3 * Ne ** 3, 2.0 * Ne ** 3
    projector = 2.0 * 2 * hl * Ne * Ne
    op = case["op"]
    if op == "energy":
        flops = moves * (S * site_wise + 2 * r * r * hl + 2 * r * hl + 2.0 / 3 * r ** 3)
        return {"bytes": B * (cache + out), "flops": B * flops}
    if op == "full":
        return {"bytes": B * (N + out) + 8 * (n_params + 2 * N * Ne), "flops": B * (moves + 1) * (forward + lu)}
    if op == "load":
        tail = lu if wide and pb.family == I.FAMILY_ACE else inverse + projector
        kept = 0 if pb.family == I.FAMILY_ACE else T * (Ne * Ne + 2 * Ne * hl + N * (h + hl))
        return {"bytes": B * (N + kept + out + 8) + T * n_params, "flops": B * (forward + tail)}
    update = 2.0 * r * Ne * (Ne + 2 * h) + 2.0 * r ** 3 + S * site_wise
    moved = 2 * T * (Ne * Ne + 2 * Ne * h)  # the inverse and the projector, read and written
    due = 1.0 / pb.refresh_every
    if op == "commit":
        return {"bytes": B * (2 * moved + 2 * (out + 4) + 16 + N), "flops": 2 * B * (update + due * (forward + inverse))}
    if op == "sweep":
        steps, rate = case["steps"], 0.3
        ratio = S * site_wise + 2 * r * r * h + 2 * Ne * r + 2.0 / 3 * r ** 3
        return {"bytes": B * (moved + 16 * steps + N + out + 8),
                "flops": B * steps * (ratio + rate * (update + due * (forward + inverse)))}
    if op == "symmetry":
        G = (pb.Lx // case["stride"]) * (pb.Ly // case["stride"])
        return {"bytes": B * (N + out + 4) + G * (8 * N + 8), "flops": B * G * (forward + lu)}
    backward = N * sum(layer) * 3 + 2 * 2.0 * Ne * Ne * h
    flops = B * (backward if op == "grad" else backward + forward + inverse + projector)
    return {"bytes": B * (out * n_params + (T * Ne * Ne if op == "grad" else N)), "flops": flops}


# ---- the same results in 64 bits, in plain torch ---------------------------------------------
class _Model64:
    def __init__(self, pb, params, M0):
        self.pb, self.M0 = pb, M0
        p = {k: params[o:o + math.prod(s)].view(s) for k, (o, s) in I.param_offsets(pb).items()}
        self.p, self.act = p, torch.tanh if pb.act == I.ACT_TANH else torch.nn.functional.silu
        self.E = p["embed"] if pb.per_site_embed else p["embed"].expand(pb.N, 4, pb.h)
        taps = [I.stencil_taps(int(k), pb.stencil) for k in pb.ksize]
        self.nbr = [torch.tensor([[_site(pb, i, dx, dy) % (pb.N + 1) for dx, dy in t] for i in range(pb.N)], device="cuda")
                    for t in taps]  # past an open edge: row N, zeros
        self.K = [p[f"kernel{l}"].reshape(len(t), *I.layer_widths(pb, l)) for l, t in enumerate(taps)]
        self.b = [p[f"bias{l}"] for l in range(pb.n_layers)]
        self.w, self.pb_ = p["proj_w"], p["proj_b"]

    def rows(self, l, x):
        """The layer's input patches [B][N][taps * c_in]."""
        x = torch.cat([x, x.new_zeros(x.shape[0], 1, x.shape[2])], 1)
        return x[:, self.nbr[l]].flatten(2)

    def features(self, occ, tape=None):
        x = self.E[torch.arange(self.pb.N, device="cuda"), occ.long()]
        if tape is not None:
            x = x.detach().requires_grad_()
            tape.append((x, None))
        for l in range(self.pb.n_layers):
            u = self.rows(l, x)
            z = u @ self.K[l].flatten(0, 1) + self.b[l]
            if tape is not None:
                tape.append((u.detach(), z))
            x = x + self.act(z) if self.pb.residual[l] else self.act(z)
            if f"ln_gamma{l}" in self.p:
                x = torch.nn.functional.layer_norm(x, x.shape[-1:], self.p[f"ln_gamma{l}"], self.p[f"ln_beta{l}"], self.pb.ln_eps)
        return x

    def slater(self, occ, H):
        """Slater matrices in ascending orbital order; the occupied orbitals."""
        pb, out, orbs = self.pb, [], []
        for s, n in ((0, pb.n_up), (1, pb.n_dn)):
            sites = (occ >> s & 1).nonzero()[:, 1].view(-1, n)
            rows = H.gather(1, sites[:, :, None].expand(-1, -1, H.shape[2]))
            cols = slice(s * pb.Ne, (s + 1) * pb.Ne)
            out.append(self.M0[s * pb.N + sites] + self.pb_[cols] + rows @ self.w[:, cols])
            orbs.append(sites + s * pb.N)
        return torch.cat(out, 1), torch.cat(orbs, 1)

    def log_psi(self, occ):
        per = max(1, int(2e8 // (self.pb.N * self.K[0].shape[0] * self.K[0].shape[1] + 2 * self.pb.Ne ** 2)))
        got = [torch.linalg.slogdet(self.slater(o, self.features(o))[0]) for o in occ.split(per)]
        return torch.cat([g[1] for g in got]), torch.cat([g[0] for g in got])

    def gradient(self, occ):
        """d log|psi| / d theta per sample: dz of every layer by autograd, the rest by products."""
        parts, pb = [], self.pb
        for o in occ.split(max(1, int(1e8 // (pb.N * self.K[0].shape[0] * pb.h * pb.n_layers)))):
            tape = []
            H = self.features(o, tape)
            Phi, orbs = self.slater(o, H)
            la = torch.linalg.slogdet(Phi)[1].sum()
            gE, *gz = torch.autograd.grad(la, [tape[0][0]] + [z for _, z in tape[1:]])
            inv_t = torch.linalg.inv(Phi.detach()).transpose(1, 2)  # d log|det| / d Phi
            n = len(o)
            g_embed = torch.zeros(n, pb.N, 4, pb.h, dtype=torch.float64, device="cuda")
            g_embed.scatter_(2, o.long()[:, :, None, None].expand(-1, -1, 1, pb.h), gE.unsqueeze(2))
            cols = [g_embed if pb.per_site_embed else g_embed.sum(1)]
            for (u, _), dz in zip(tape[1:], gz):
                cols += [u.transpose(1, 2) @ dz, dz.sum(1)]
            Hr = H.detach().gather(1, (orbs % pb.N)[:, :, None].expand(-1, -1, H.shape[2]))
            by_spin = [(Hr[:, a:b], inv_t[:, a:b]) for a, b in ((0, pb.n_up), (pb.n_up, pb.Ne))]
            cols += [torch.cat([x.transpose(1, 2) @ g for x, g in by_spin], 2), torch.cat([g.sum(1) for _, g in by_spin], 1)]
            parts.append(torch.cat([c.reshape(n, -1) for c in cols], 1))
        return torch.cat(parts)

    def local_energy(self, occ):
        """sum over n' of <n|H|n'> psi(n')/psi(n), each ratio a determinant over the electrons on
        the sites whose features the move changes (the layers after the first are site-wise)."""
        pb, N, Ne = self.pb, self.pb.N, self.pb.Ne
        nn, nnn = _bonds(pb)
        bonds = torch.tensor(nn + nnn, device="cuda")
        sees = [[] for _ in range(N + 1)]  # the sites whose first layer reads site t
        for i, row in enumerate(self.nbr[0].tolist()):
            for t in row:
                sees[t].append(i)
        S = [sorted(set(sees[i] + sees[j])) for i, j in nn + nnn]
        width = max(len(x) for x in S)
        S = torch.tensor([x + [-1] * (width - len(x)) for x in S], device="cuda")
        KE = torch.einsum("inc,dce->inde", self.E, self.K[0])  # layer-0 response to a state on a site
        KE = torch.cat([KE, KE.new_zeros(1, *KE.shape[1:])])
        M0b = self.M0 + self.pb_.view(2, 1, Ne).expand(2, N, Ne).reshape(2 * N, Ne)
        W = self.w.view(-1, 2, Ne).transpose(0, 1)
        up, dn = occ & 1, occ >> 1 & 1
        if pb.model == I.MODEL_TJ:
            sz = (up - dn).double()
            energy = pb.J / 4 * (sz[:, bonds[:len(nn), 0]] * sz[:, bonds[:len(nn), 1]]).sum(1)
        else:
            energy = pb.U * (up * dn if pb.model == I.MODEL_HUBBARD else up * (1 - dn)).sum(1).double()
        for at in torch.arange(len(occ), device="cuda").split(max(1, int(3e8 // (Ne * Ne + N * pb.h * 13)))):
            o = occ[at]
            Phi, _ = self.slater(o, self.features(o))
            inv_t = torch.linalg.inv(Phi).transpose(1, 2).contiguous()
            bits = torch.cat([o & 1, o >> 1 & 1], 1)
            slot = bits.cumsum(1) - 1
            oi, oj = o[:, bonds[:, 0]], o[:, bonds[:, 1]]
            lists = []  # (walker, bond, new states of the two sites, matrix element)
            t = torch.tensor([pb.t] * len(nn) + [pb.tp] * len(nnn), dtype=torch.float64, device="cuda")
            for s in (0, 1):
                hi, hj = oi >> s & 1, oj >> s & 1
                ok = hi != hj
                if pb.model == I.MODEL_TJ:
                    ok &= (oi == 0) | (oj == 0)
                w, q = ok.nonzero(as_tuple=True)
                lists.append((w, q, oi[w, q] ^ 1 << s, oj[w, q] ^ 1 << s, -t[q]))
            if pb.model == I.MODEL_TJ and pb.J:
                w, q = (((oi == 1) & (oj == 2)) | ((oi == 2) & (oj == 1)))[:, :len(nn)].nonzero(as_tuple=True)
                lists.append((w, q, oj[w, q], oi[w, q], torch.full((len(w),), -pb.J / 2, dtype=torch.float64, device="cuda")))
            w, q, ni, nj, coeff = (torch.cat(x) for x in zip(*lists))
            per = max(1, int(2.5e8 // (width * max(self.K[0].shape[0] * pb.h, 4 * Ne, max(k.shape[2] for k in self.K) * 4))))
            for m in torch.arange(len(w), device="cuda").split(per):
                wm, (i, j) = w[m], bonds[q[m]].T
                new = o[wm].clone()
                k = torch.arange(len(m), device="cuda")
                new[k, i], new[k, j] = ni[m], nj[m]
                Sm = S[q[m]]
                site = Sm.clamp(min=0)
                near = self.nbr[0][site]
                state = torch.cat([new, new.new_zeros(len(m), 1)], 1)[k[:, None, None], near].long()
                z = self.b[0].expand(len(m), width, -1).clone()
                for d in range(near.shape[2]):
                    z += KE[near[:, :, d], state[:, :, d], d]
                x = self.act(z) + (self.E[site, new[k[:, None], site].long()] if pb.residual[0] else 0)
                for l in range(1, pb.n_layers):
                    y = self.act(x @ self.K[l][0] + self.b[l])
                    x = x + y if pb.residual[l] else y
                orb = torch.cat([site, site + N], 1)
                there = torch.cat([new[k[:, None], site] & 1, new[k[:, None], site] >> 1 & 1], 1).bool() & torch.cat([Sm, Sm], 1).ge(0)
                other = torch.where(site == i[:, None], j[:, None], i[:, None])  # where a moved electron came from
                before = torch.where(bits[wm].gather(1, orb).bool(), orb, torch.cat([other, other + N], 1))
                c = torch.where(there, slot[wm].gather(1, before), 0)
                rows = M0b[orb] + torch.cat([x @ W[0], x @ W[1]], 1)
                R = rows @ inv_t[wm[:, None], c].transpose(1, 2)
                R = torch.where(there[:, :, None] & there[:, None, :], R, torch.eye(R.shape[1], dtype=R.dtype, device="cuda"))
                energy.index_add_(0, at[wm], coeff[m] * torch.linalg.det(R))
        return energy


def _parity(perm, occ, orbs):
    """Sign of the permutation sorting the images of the occupied orbitals."""
    img = perm[orbs]
    swapped = (img[:, :, None] > img[:, None, :]).triu(1).sum((1, 2))
    return 1.0 - 2.0 * (swapped % 2).double()


def exact(case, seed):
    op = case["op"]
    if op == "sweep":
        return None
    pb, params, M0, occ, gen = _inputs(case, seed)
    m = _Model64(pb, params, M0)
    if op in ("energy", "full"):
        return m.local_energy(occ)
    if op == "load":
        return m.log_psi(occ)[0], None, None
    if op == "commit":
        there, _ = _accepted_moves(pb, M0, occ, gen)
        new, k = occ.clone(), torch.arange(len(occ), device="cuda")
        src, dst, bit = there[:, 1].long(), there[:, 2].long(), (1 << there[:, 3]).to(torch.int8)
        new[k, src] ^= bit
        new[k, dst] ^= bit
        return m.log_psi(new)[0], None, m.log_psi(occ)[0], None, None
    if op == "symmetry":
        orbs = torch.cat([(occ & 1), (occ >> 1 & 1)], 1).nonzero()[:, 1].view(len(occ), pb.Ne)
        logs, signs = [], []
        for perm in _group(pb, case["stride"]).long():
            image = torch.zeros_like(occ)
            image[:, perm[:pb.N]] = occ  # a translation moves both spins of a site alike
            la, sg = m.log_psi(image)
            logs.append(la)
            signs.append(sg * _parity(perm, occ, orbs))
        la, sg = torch.stack(logs), torch.stack(signs)
        top = la.max(0).values
        return top + (sg * (la - top).exp()).sum(0).abs().log(), None
    return m.gradient(occ)
