"""The work that is timed: passes through the public entry points, over the ranges they are used in.

A case names an entry point (``kind``), an angular-momentum class (``cls``, the l of the shells in order, e.g. "2120"
for (dp|ds)), the primitives per shell (``K``; 0: the mixed degrees 6, 3 and 1 of a molecular basis), the lists' lengths
and the exponents (``exps``).  Shells sit in a 12-bohr cube, each on a centre of its own; contraction coefficients are
weights U[0.5, 1] times the usual normalisation.  ``exact`` is an independent McMurchie-Davidson evaluation in 64-bit
torch: dense Hermite tables, no recursion forms, no sorting.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2506_12501_gb300 as eri

CUBE = 12.0
RACAH = {  # real solid harmonics, m = -l..l: (coefficient, x power, y power, z power)
    0: [[(1.0, 0, 0, 0)]],
    1: [[(1.0, 0, 1, 0)], [(1.0, 0, 0, 1)], [(1.0, 1, 0, 0)]],
    2: [[(3 ** 0.5, 1, 1, 0)], [(3 ** 0.5, 0, 1, 1)], [(-0.5, 2, 0, 0), (-0.5, 0, 2, 0), (1.0, 0, 0, 2)],
        [(3 ** 0.5, 1, 0, 1)], [(0.75 ** 0.5, 2, 0, 0), (-(0.75 ** 0.5), 0, 2, 0)]],
    3: [[(3 * 0.625 ** 0.5, 2, 1, 0), (-(0.625 ** 0.5), 0, 3, 0)], [(15 ** 0.5, 1, 1, 1)],
        [(4 * 0.375 ** 0.5, 0, 1, 2), (-(0.375 ** 0.5), 2, 1, 0), (-(0.375 ** 0.5), 0, 3, 0)],
        [(1.0, 0, 0, 3), (-1.5, 2, 0, 1), (-1.5, 0, 2, 1)],
        [(4 * 0.375 ** 0.5, 1, 0, 2), (-(0.375 ** 0.5), 3, 0, 0), (-(0.375 ** 0.5), 1, 2, 0)],
        [(3.75 ** 0.5, 2, 0, 1), (-(3.75 ** 0.5), 0, 2, 1)],
        [(0.625 ** 0.5, 3, 0, 0), (-3 * 0.625 ** 0.5, 1, 2, 0)]],
}


# ---------------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------------
def _batch(kind, cls, K, npairs, nq, exps="even", **more):
    """npairs shell pairs on each side; nq > 0: that many random quartets of them, 0: every combination."""
    return dict(kind=kind, cls=cls, K=K, npairs=npairs, nket=npairs, nq=nq, exps=exps, **more)


def listed():
    return [
        # the smallest call: 1000 quartets of uncontracted p shells, where launches and latency are all
        dict(name="pp_pp_small", **_batch("fwd", "1111", 1, 1000, 1000, "free")),
        # the lightest class over a molecular basis: s shells of 6, 3 and 1 primitives in one list
        dict(name="ss_ss_mixed", **_batch("fwd", "0000", 0, 2048, 400_000)),
        # an ordinary class of a contracted sp basis
        dict(name="pp_ps", **_batch("fwd", "1110", 3, 2048, 100_000)),
        # every combination of a bra and a ket list of odd lengths, as a driver over shell-pair blocks calls it
        dict(name="dp_pp_blocks", kind="fwd", cls="2111", K=3, npairs=211, nket=307, nq=0, exps="even"),
        # the heaviest class of a polarised double-zeta basis
        dict(name="dd_dd", **_batch("fwd", "2222", 3, 2048, 30_000)),
        # uncontracted f shells of a polarised triple-zeta basis
        dict(name="ff_dd_uncontracted", **_batch("fwd", "3322", 1, 2048, 20_000, "wide")),
        # high angular momentum with contraction, in the split precision the caller may choose
        dict(name="ff_dd_split", **_batch("split", "3322", 3, 1024, 4_000, "wide")),
        # solid-harmonic output, as most basis sets want it
        dict(name="dd_dp_sph", **_batch("sph", "2221", 3, 1024, 20_000)),
        # density fitting: solid-harmonic auxiliary shells (uncontracted) against orbital pairs
        dict(name="f_dp_three_centre", **_batch("three", "3021", 3, 2048, 100_000, pure=True)),
        # nuclear and exponent gradients over a molecular basis (mixed degrees)
        dict(name="ps_ps_gradient", **_batch("grad", "1010", 0, 1024, 60_000)),
        # a differentiable forward and its backward, as an optimisation of a basis or geometry runs them
        dict(name="dp_pp_training", **_batch("train", "2111", 3, 512, 6_000)),
        # Coulomb and exchange matrices of a whole molecule, one Fock build
        dict(name="molecule_jk", kind="plan", natom=12, radius=4.0, threshold=1e-12),
    ]


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["fwd", "fwd", "fwd", "split", "sph", "three", "grad", "train", "plan"])
        if kind == "plan":
            natom = rng.randint(4, 11)
            return dict(kind=kind, natom=natom, radius=round(4.0 * (natom / 12) ** (1 / 3) * rng.uniform(0.97, 1.1), 3),
                        threshold=rng.choice([1e-12, 1e-11, 1e-10]))
        high = kind in ("fwd", "split", "sph") and rng.random() < 0.25
        l = [rng.randint(0, 3 if high else 2) for _ in range(4)]
        if kind in ("grad", "train"):
            l = [min(x, rng.choice([1, 1, 2])) for x in l]
        K = rng.choice([1, 2, 3, 3, 4]) if kind not in ("grad", "train") else rng.choice([1, 2, 3])
        exps = rng.choice(["even", "even", "wide", "free"])
        if max(l) == 0 and exps == "even" and kind in ("fwd", "grad"):
            K = 0
        if sum(l) > 8 and K > 3:
            continue
        if kind == "three":
            l[0], l[1] = rng.randint(0, 3), 0
        npairs, nket = (round(math.exp(rng.uniform(math.log(40), math.log(3000)))) for _ in range(2))
        top = {"grad": 60_000, "train": 20_000, "split": 20_000}.get(kind, 400_000)
        nq = round(math.exp(rng.uniform(math.log(200), math.log(top))))
        if kind == "fwd" and rng.random() < 0.25 and npairs * nket <= 400_000:
            nq = 0
        case = dict(kind=kind, cls="".join(map(str, l)), K=K, npairs=npairs, nket=nket, nq=nq, exps=exps)
        if kind == "three":
            case["pure"] = rng.random() < 0.6
        weight = {"grad": 6, "train": 8}.get(kind, 1)
        if weight * work(case)["flops"] <= 0.8 * most:
            return case


# ---------------------------------------------------------------------------------------------------------------------
# sizes and operation counts
# ---------------------------------------------------------------------------------------------------------------------
def nc(l):
    return (l + 1) * (l + 2) // 2


def nh(l):
    return (l + 1) * (l + 2) * (l + 3) // 6


@functools.lru_cache(None)
def carts(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


@functools.lru_cache(None)
def hermites(L):
    return [(t, u, N - t - u) for N in range(L + 1) for t in range(N, -1, -1) for u in range(N - t, -1, -1)]


def _terms(l1, l2):
    """Non-zero Hermite terms of the (e0| functions a shell pair needs (the pair follows by horizontal recursion)."""
    return sum((e[0] + 1) * (e[1] + 1) * (e[2] + 1) for l in range(l1, l1 + l2 + 1) for e in carts(l))


def _degrees(case):
    """Mean K_a K_b of a pair (mixed degrees: of 6, 3, 1)."""
    k = 10 / 3 if case["K"] == 0 else case["K"]
    return k * k


def _class(case):
    return tuple(int(c) for c in case["cls"])


def _quartet_flops(cls, kb, kk):
    la, lb, lc, ld = cls
    L = la + lb + lc + ld
    aux = 40 + 5 * L + 2 * (math.comb(L + 4, 4) - L - 1)          # Boys, prefactors, auxiliary recursion
    cols = sum(nc(l) for l in range(lc, lc + ld + 1))
    a = kb * kk * 2 * nh(la + lb) * _terms(lc, ld) + kb * 2 * cols * _terms(la, lb)
    rows = sum(nc(l) for l in range(la, la + lb + 1))
    b = kb * kk * 2 * nh(lc + ld) * _terms(la, lb) + kk * 2 * rows * _terms(lc, ld)
    return kb * kk * aux + min(a, b)


def work(case):
    if case["kind"] == "plan":
        nat, deg = case["natom"], {0: (6, 3, 1), 1: (3, 1), 2: (1,)}
        nbf = 15 * nat
        pairs = [(l1, l2, k1 * k2) for l1 in deg for k1 in deg[l1] for l2 in deg if l2 <= l1 for k2 in deg[l2]]
        n = nat * nat
        fl = sum(0.5 * n * n * 0.5 * (_quartet_flops((a, b, c, d), k, m) + 4 * nc(a) * nc(b) * nc(c) * nc(d) * 3)
                 for a, b, k in pairs for c, d, m in pairs) / 2
        return {"bytes": 8.0 * 3 * nbf * nbf, "flops": float(fl)}
    cls, pp = _class(case), _degrees(case)
    kx = 1 if case["kind"] == "three" else pp
    nq = case["nq"] or case["npairs"] * case["nket"]
    n_out = math.prod(2 * l + 1 if case["kind"] == "sph" else nc(l) for l in cls)
    if case["kind"] == "three" and case["pure"]:
        n_out = (2 * cls[0] + 1) * nc(cls[2]) * nc(cls[3])
    fl = nq * _quartet_flops(cls, kx, pp)
    by = 8.0 * nq * n_out + 16.0 * case["nq"] + 8.0 * (case["npairs"] + case["nket"])
    if case["kind"] in ("grad", "train"):  # the derivatives of E in centres and exponents: both sides raised by two
        la, lb, lc, ld = cls
        raised = nq * (pp * pp * (40 + 5 * sum(cls) + 2 * math.comb(sum(cls) + 6, 4) +
                                  2 * nh(la + lb + 2) * _terms(lc, ld) + 2 * nh(lc + ld + 2) * _terms(la, lb)) +
                       2 * pp * n_out * 20)
        fl = raised + (fl if case["kind"] == "train" else 0)
        by += 8.0 * nq * n_out if case["kind"] == "train" else 0.0
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    """About four times what the paths show against ``exact``: up to 3.4e-14 with FP64 transforms (where the recursion
    forms magnify rounding; 2e-15 without them), 1e-13 with split ones, 7e-15 for gradients, 2.5e-15 for J and K, whose
    screened quartets add differences of the threshold's size."""
    if case["kind"] == "plan":
        return {"rel": 1e-13 * max(1.0, case["threshold"] / 1e-12)}
    if case["kind"] == "grad":
        return {"rel": 3e-14}
    return {"rel": 4e-13 if case["kind"] == "split" else 1.5e-13}


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
def _norm(z, l):
    return (2 * z / math.pi) ** 0.75 * (4 * z) ** (0.5 * l) / math.sqrt(math.prod(range(2 * l - 1, 0, -2)))


def _shell(rng, l, K, exps):
    if exps == "even":      # even-tempered, the same for every shell
        z = 0.2 * 3.0 ** np.arange(K)
    elif exps == "wide":
        z = 10.0 ** rng.uniform(math.log10(0.05), math.log10(50.0), K)
    else:                   # "free"
        z = 10.0 ** rng.uniform(-1.0, 1.0, K)
    return z, rng.uniform(0.5, 1.0, K) * _norm(z, l)


def _basis(centres, shells):
    """shells: (atom, l, exponents, coefficients); the layout DeviceBasis takes."""
    K = np.array([len(s[2]) for s in shells], np.int32)
    return dict(centres=np.asarray(centres, np.float64), shell_atom=np.array([s[0] for s in shells], np.int32),
                shell_l=np.array([s[1] for s in shells], np.int32), shell_K=K,
                shell_off=np.concatenate([[0], np.cumsum(K)[:-1]]).astype(np.int32),
                exps=np.concatenate([s[2] for s in shells]), coefs=np.concatenate([s[3] for s in shells]))


def _inputs(case, seed):
    """Basis, bra list, ket list, quartets (None: every combination) and weights, as numpy arrays."""
    rng = np.random.default_rng([seed, 11])
    cls, pool = _class(case), min(512, 2 * max(case["npairs"], case["nket"]))
    shells, start = [], {}
    for i, l in enumerate(cls):
        aux = case["kind"] == "three" and i == 0
        start[i] = len(shells)
        for j in range(pool):
            K = 1 if aux else (case["K"] or (6, 3, 1)[j % 3])
            shells.append((len(shells), l) + _shell(rng, l, K, "free" if aux else case["exps"]))
    basis = _basis(rng.uniform(0.0, CUBE, (len(shells), 3)), shells)
    pick = [start[i] + rng.integers(0, pool, case["npairs"] if i < 2 else case["nket"]) for i in range(4)]
    bra = np.stack(pick[:2], 1).astype(np.int32)
    ket = np.stack(pick[2:], 1).astype(np.int32)
    if case["kind"] == "three":
        bra = bra[:, 0].copy()
    quartets = None
    if case["nq"]:
        quartets = np.stack([rng.integers(0, case["npairs"], case["nq"]), rng.integers(0, case["nket"], case["nq"])],
                            1).astype(np.int64)
    nq = case["nq"] or case["npairs"] * case["nket"]
    W = None
    if case["kind"] in ("grad", "train"):
        W = rng.uniform(-1.0, 1.0, nq * math.prod(nc(l) for l in cls))
    return basis, bra, ket, quartets, W


def _molecule(case, seed):
    """Atoms in a sphere at least 1.8 bohr apart, each with s (6, 3, 1 primitives), p (3, 1) and d (1) shells."""
    rng = np.random.default_rng([seed, 12])
    pts = []
    while len(pts) < case["natom"]:
        p = rng.uniform(-case["radius"], case["radius"], 3)
        if p @ p <= case["radius"] ** 2 and all(np.linalg.norm(p - q) >= 1.8 for q in pts):
            pts.append(p)
    shells = [(a, l) + _shell(rng, l, K, "even") for a in range(len(pts))
              for l, K in ((0, 6), (0, 3), (0, 1), (1, 3), (1, 1), (2, 1))]
    basis = _basis(np.array(pts), shells)
    nbf = int(sum(nc(l) for l in basis["shell_l"]))
    U = rng.uniform(-1.0, 1.0, (nbf, nbf))
    return basis, np.triu(U) + np.triu(U, 1).T


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "plan":
        basis, D = _molecule(case, seed)
        db = eri.DeviceBasis(basis)
        D = torch.as_tensor(D, device=dev)
        return dict(case=case, db=db, plan=eri.Plan(db, case["threshold"]), D=D, J=torch.empty_like(D),
                    K=torch.empty_like(D))
    basis, bra, ket, quartets, W = _inputs(case, seed)
    s = dict(case=case, cls=_class(case), db=eri.DeviceBasis(basis), bra=torch.as_tensor(bra, device=dev),
             ket=torch.as_tensor(ket, device=dev),
             quartets=None if quartets is None else torch.as_tensor(quartets, device=dev))
    if W is not None:
        s["W"] = torch.as_tensor(W, device=dev)
    if case["kind"] == "train":
        s["centres"] = s["db"].centres.clone().requires_grad_()
        s["exps"] = s["db"].exps.clone().requires_grad_()
    return s


def run(state):
    kind, s = state["case"]["kind"], state
    if kind == "plan":
        return list(s["plan"].jk(s["D"], J=s["J"], K=s["K"]))
    if kind == "sph":
        return eri.eri_batch_sph(s["cls"], s["db"], s["bra"], s["ket"], s["quartets"])
    if kind == "three":
        lx, _, lc, ld = s["cls"]
        return eri.eri_batch3(lx, lc, ld, s["db"], s["bra"], s["ket"], s["quartets"], pure=s["case"]["pure"])
    if kind == "grad":
        gc, ge = torch.zeros_like(s["db"].centres), torch.zeros_like(s["db"].exps)
        return list(eri.eri_batch_grad(s["cls"], s["db"], s["bra"], s["ket"], s["quartets"], s["W"], gc, ge))
    if kind == "train":
        out = eri.eri(s["centres"], s["exps"], s["cls"], s["db"], s["bra"], s["ket"], s["quartets"])
        gc, ge = torch.autograd.grad((out * s["W"]).sum(), (s["centres"], s["exps"]))
        return [out.detach(), gc, ge]
    precision = eri.ERI_PREC_SPLIT if kind == "split" else eri.ERI_PREC_FP64
    return eri.eri_batch(s["cls"], s["db"], s["bra"], s["ket"], s["quartets"], precision=precision)


# ---------------------------------------------------------------------------------------------------------------------
# the same integrals in plain 64-bit torch
# ---------------------------------------------------------------------------------------------------------------------
class _Boys(torch.autograd.Function):
    """F_0..F_L at T, [L+1, ...]; dF_m/dT = -F_{m+1}."""

    @staticmethod
    def forward(ctx, T, L):
        top = L + 1 if T.requires_grad else L
        small = T < 36.0
        t = torch.where(small, T, torch.full_like(T, 36.0))
        eT, term = torch.exp(-t), torch.full_like(t, 1.0 / (2 * top + 1))
        acc = term.clone()
        for k in range(1, 190):
            term = term * (2 * t / (2 * top + 2 * k + 1))
            acc = acc + term
        lo = [None] * (top + 1)
        lo[top] = eT * acc
        for m in range(top - 1, -1, -1):
            lo[m] = (2 * t * lo[m + 1] + eT) / (2 * m + 1)
        t = torch.where(small, torch.full_like(T, 36.0), T)
        eT, hi = torch.exp(-t), [0.5 * torch.sqrt(math.pi / t) * torch.erf(torch.sqrt(t))]
        for m in range(top):
            hi.append(((2 * m + 1) * hi[m] - eT) / (2 * t))
        F = torch.stack([torch.where(small, a, b) for a, b in zip(lo, hi)])
        if T.requires_grad:
            ctx.save_for_backward(F)
        return F[:L + 1]

    @staticmethod
    def backward(ctx, g):
        (F,) = ctx.saved_tensors
        return -(g * F[1:]).sum(0), None


def _aux(L, T, rho, pref, d):
    """[tuv]^(0), |tuv| <= L, as a list in the order of ``hermites(L)``; d: the three components of P - Q."""
    F = _Boys.apply(T, L)
    idx = {h: i for i, h in enumerate(hermites(L))}
    cur = None
    for n in range(L, -1, -1):
        base = pref * (-2.0 * rho) ** n * F[n]
        new = [base]
        for h in hermites(L - n)[1:]:
            i = min((a for a in range(3) if h[a]), key=lambda a: h[a])
            h1 = tuple(h[a] - (a == i) for a in range(3))
            v = d[i] * cur[idx[h1]]
            if h[i] > 1:
                h2 = tuple(h[a] - 2 * (a == i) for a in range(3))
                v = v + (h[i] - 1) * cur[idx[h2]]
            new.append(v)
        cur = new
    return cur


def _pair(l1, l2, A, B, za, zb, ca, cb):
    """Pair exponents [n, k], centres [n, k, 3] and dense expansion coefficients [n, k, Hermite, component pair]."""
    n = za.shape[0]
    za, zb = (x.reshape(n, -1) for x in torch.broadcast_tensors(za[:, :, None], zb[:, None, :]))
    c = (ca[:, :, None] * cb[:, None, :]).reshape(n, -1)
    p = za + zb
    P = (za[..., None] * A[:, None] + zb[..., None] * B[:, None]) / p[..., None]
    ax = []
    for i in range(3):
        PA, PB, h = P[..., i] - A[:, None, i], P[..., i] - B[:, None, i], 0.5 / p
        E = {(0, 0, 0): torch.exp(-za * zb / p * ((A - B)[:, None, i]) ** 2)}

        def get(a, b, t):
            return E.get((a, b, t))

        for a in range(l1 + 1):
            for b in range(l2 + 1):
                if a + b == 0:
                    continue
                src, X = ((a - 1, b), PA) if a else ((a, b - 1), PB)
                for t in range(a + b + 1):
                    v = 0.0
                    if get(*src, t - 1) is not None:
                        v = v + h * get(*src, t - 1)
                    if get(*src, t) is not None:
                        v = v + X * get(*src, t)
                    if get(*src, t + 1) is not None:
                        v = v + (t + 1) * get(*src, t + 1)
                    E[a, b, t] = v
        ax.append(E)
    zero = torch.zeros_like(p)
    rows = []
    for h in hermites(l1 + l2):
        for x in carts(l1):
            for y in carts(l2):
                e = [ax[i].get((x[i], y[i], h[i])) for i in range(3)]
                rows.append(zero if any(f is None for f in e) else c * e[0] * e[1] * e[2])
    M = torch.stack(rows, -1).reshape(n, p.shape[1], nh(l1 + l2), nc(l1) * nc(l2))
    return p, P, M


def _integrals(cls, bra, ket):
    """(ab|cd) [n, ab, cd] of n quartets from their two sides' pair data (see ``_pair``)."""
    la, lb, lc, ld = cls
    (p, P, Eb), (q, Q, Ek) = bra, ket
    p, q = p[:, :, None], q[:, None, :]
    rho = p * q / (p + q)
    d = P[:, :, None] - Q[:, None, :]
    pref = 2.0 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q))
    R = torch.stack(_aux(sum(cls), rho * (d * d).sum(-1), rho, pref, d.unbind(-1)), -1)    # [n, i, k, tuv]
    idx = {h: i for i, h in enumerate(hermites(sum(cls)))}
    hb, hk = hermites(la + lb), hermites(lc + ld)
    pq = torch.tensor([[idx[tuple(a + b for a, b in zip(x, y))] for y in hk] for x in hb], device=p.device)
    sign = torch.tensor([(-1.0) ** sum(y) for y in hk], dtype=torch.float64, device=p.device)
    n, nb, nk = R.shape[:3]
    G = R.index_select(3, pq.reshape(-1)).reshape(n, nb, nk, len(hb), len(hk))
    X = torch.bmm(G.permute(0, 1, 3, 2, 4).reshape(n, nb * len(hb), nk * len(hk)),
                  (Ek * sign[:, None]).reshape(n, nk * len(hk), -1))
    return torch.bmm(Eb.reshape(n, nb * len(hb), -1).transpose(1, 2), X)


def _solid(l, dev):
    M = torch.zeros(2 * l + 1, nc(l), dtype=torch.float64, device=dev)
    for m, row in enumerate(RACAH[l]):
        for c, x, y, z in row:
            M[m, carts(l).index((x, y, z))] += c
    return M


class _Shells:
    """The shells' centres and zero-padded primitives on the device (differentiable in centres and exponents)."""

    def __init__(self, basis, dev, grad=False):
        t = functools.partial(torch.as_tensor, device=dev)
        self.centres, self.exps = t(basis["centres"]).requires_grad_(grad), t(basis["exps"]).requires_grad_(grad)
        K, off = basis["shell_K"], basis["shell_off"]
        slot = np.arange(K.max())[None, :]
        self.atom, self.real = t(basis["shell_atom"]).long(), t(slot < K[:, None])
        self.slot = t(np.where(slot < K[:, None], off[:, None] + slot, 0)).long()
        self.c = torch.where(self.real, t(basis["coefs"])[self.slot], torch.zeros((), dtype=torch.float64, device=dev))
        self.l = basis["shell_l"]

    def pair(self, l1, l2, i, j):
        """Pair data of the shells i and j (tensors); j None: the unit function."""
        A = self.centres[self.atom[i]]
        one = torch.ones((), dtype=torch.float64, device=A.device)
        z = [torch.where(self.real[s], self.exps[self.slot[s]], one) for s in (i, j) if s is not None]
        c = [self.c[s] for s in (i, j) if s is not None]
        k = [int(self.real[s].sum(1).max()) for s in (i, j) if s is not None]
        if j is None:
            z.append(torch.zeros(len(i), 1, dtype=torch.float64, device=A.device))
            c.append(torch.ones(len(i), 1, dtype=torch.float64, device=A.device))
            k.append(1)
        B = A if j is None else self.centres[self.atom[j]]
        return _pair(l1, l2, A, B, z[0][:, :k[0]], z[1][:, :k[1]], c[0][:, :k[0]], c[1][:, :k[1]])


def _chunk(cls, prims):
    """Quartets evaluated at once: about 4 GB of intermediates."""
    doubles = prims * (nh(sum(cls)) * 3 + nh(cls[0] + cls[1]) * nh(cls[2] + cls[3]) * 2)
    return max(1, int(5e8 / doubles))


def _exact_batch(case, seed, dev):
    basis, bra, ket, quartets, W = _inputs(case, seed)
    cls, kind = _class(case), case["kind"]
    grad = kind in ("grad", "train")
    if quartets is None:
        q = np.arange(case["npairs"] * case["nket"])
        quartets = np.stack([q % case["npairs"], q // case["npairs"]], 1)
    sh, nq = _Shells(basis, dev, grad), len(quartets)
    sides = []
    for l1, l2, lst, col in ((cls[0], cls[1], bra, 0), (cls[2], cls[3], ket, 1)):
        lst = torch.as_tensor(lst.reshape(len(lst), -1), device=dev).long()
        sides.append((l1, l2, lst[:, 0], lst[:, 1] if lst.shape[1] == 2 else None,
                      torch.as_tensor(quartets[:, col], device=dev)))
    kmax = (case["K"] or 6) ** 2
    step = _chunk(cls, kmax * kmax) // (6 if grad else 1)
    out = torch.empty(nq, nc(cls[0]) * nc(cls[1]), nc(cls[2]) * nc(cls[3]), dtype=torch.float64, device=dev)
    if W is not None:
        Wt = torch.as_tensor(W, device=dev).reshape(-1, nq).T.reshape(out.shape)
    gc, ge = torch.zeros_like(sh.centres), torch.zeros_like(sh.exps)
    for s in range(0, nq, max(1, step)):
        e = min(nq, s + max(1, step))
        v = _integrals(cls, *(sh.pair(l1, l2, i[x[s:e]], None if j is None else j[x[s:e]]) for l1, l2, i, j, x in sides))
        out[s:e] = v.detach()
        if grad:
            a, b = torch.autograd.grad((v * Wt[s:e]).sum(), (sh.centres, sh.exps))
            gc, ge = gc + a, ge + b
    if kind == "sph" or (kind == "three" and case["pure"]):
        M = [_solid(l, dev) if kind == "sph" or i == 0 else torch.eye(nc(l), dtype=torch.float64, device=dev)
             for i, l in enumerate(cls)]
        out = torch.einsum("ia,jb,kc,ld,nabcd->nijkl", *M, out.reshape(nq, *(nc(l) for l in cls)))
        out = out.reshape(nq, M[0].shape[0] * M[1].shape[0], -1)
    if case["nq"]:
        flat = out.permute(1, 2, 0).reshape(-1)                                  # [ab, cd, quartet]
    else:
        flat = out.reshape(case["nket"], case["npairs"], *out.shape[1:]).permute(0, 3, 2, 1).reshape(-1)
    if kind == "train":
        return [flat, gc, ge]
    return [gc, ge] if kind == "grad" else flat


def _exact_plan(case, seed, dev):
    """J and K from the whole tensor (uv|ls), assembled class by class."""
    basis, D = _molecule(case, seed)
    sh, l = _Shells(basis, dev), basis["shell_l"]
    n = np.array([nc(x) for x in l])
    off = np.concatenate([[0], np.cumsum(n)])
    nbf = int(off[-1])
    T = torch.zeros(nbf, nbf, nbf, nbf, dtype=torch.float64, device=dev)
    i, j = np.tril_indices(len(l))
    K = basis["shell_K"]
    groups = {}
    for a, b in zip(i, j):
        a, b = (a, b) if (l[a], K[a]) >= (l[b], K[b]) else (b, a)
        groups.setdefault((int(l[a]), int(l[b]), int(K[a] * K[b])), []).append((a, b))
    groups = sorted(groups.items())
    for x, ((la, lb, kb), bra) in enumerate(groups):
        for (lc, ld, kk), ket in groups[:x + 1]:
            cls, bra_t, ket_t = (la, lb, lc, ld), np.array(bra), np.array(ket)
            total, step = len(bra) * len(ket), _chunk((la, lb, lc, ld), kb * kk)
            for s in range(0, total, step):
                q = np.arange(s, min(total, s + step))
                S = np.concatenate([bra_t[q // len(ket)], ket_t[q % len(ket)]], 1)
                P = [torch.as_tensor(S[:, c], device=dev).long() for c in range(4)]
                v = _integrals(cls, sh.pair(la, lb, P[0], P[1]), sh.pair(lc, ld, P[2], P[3]))
                v = v.reshape(len(q), *(nc(z) for z in cls))
                f = [torch.as_tensor(off[S[:, c]], device=dev)[:, None] + torch.arange(nc(cls[c]), device=dev)
                     for c in range(4)]
                a, b, c, d = (f[m].reshape(len(q), *(-1 if w == m else 1 for w in range(4))) for m in range(4))
                for u, w, g, h in ((a, b, c, d), (b, a, c, d), (a, b, d, c), (b, a, d, c)):
                    T[u, w, g, h] = v
                    T[g, h, u, w] = v
    D = torch.as_tensor(D, device=dev)
    return [torch.einsum("uvls,ls->uv", T, D), torch.einsum("uvls,vs->ul", T, D)]


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "plan":
        return _exact_plan(case, seed, dev)
    return _exact_batch(case, seed, dev)
