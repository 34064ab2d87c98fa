"""The work that a user of this package has it do, as measurable cases.

A case is one call (or one replay) of a public entry point on a molecule of
the package's own workloads: two-electron TDA gradients in fp64 and on the
routed fp32 / fp64 path, over Cartesian and spherical shells, Fock-type
builds and batches of small molecules.  ``listed`` holds the cases, ``draw``
gives more of the same ranges, ``prepare`` makes the inputs of a case from a
seed, ``run`` is one pass, ``work`` the arithmetic and traffic a pass cannot
do without, and ``exact`` the same outputs from a plain 64-bit evaluation of
the definition (small systems only).

The molecule and its basis set belong to the case.  The seed draws the
densities and displaces every atom by a few hundredths of a bohr, as from one
step of a geometry optimisation to the next.
"""
import functools
import os

import numpy as np
import torch

import paper_2407_16586_gb300 as tg
from paper_2407_16586_gb300 import synth

PRECISION = {"fp64": tg.TG_FP64, "bound": tg.TG_MIXED_BOUND, "learned": tg.TG_MIXED_LEARNED}
ROUTER = os.path.join(os.path.dirname(os.path.abspath(tg.__file__)), "data", "router.bin")


def listed():
    return [
        # one small molecule from host arrays: launches, the plan and short kernels count most
        {"name": "water-fp64", "kind": "grad", "mol": "chain", "mol_seed": 20, "nheavy": 1, "nh": 2,
         "precision": "fp64", "device": False, "rank": 0, "nranks": 1},
        # the 6-atom workload (two density pairs, one of them long-range only), plain fp64
        {"name": "c1-fp64", "kind": "grad", "mol": "config", "mol_seed": 0, "nheavy": 2, "nh": 4,
         "precision": "fp64", "device": False, "rank": 0, "nranks": 1},
        # the same molecule on the learned fp32 / fp64 route
        {"name": "c1-learned", "kind": "grad", "mol": "config", "mol_seed": 0, "nheavy": 2, "nh": 4,
         "precision": "learned", "device": False, "rank": 0, "nranks": 1},
        # an ordinary 12-atom molecule, densities resident on the GPU as in an SCF program
        {"name": "chain12-fp64", "kind": "grad", "mol": "chain", "mol_seed": 12, "nheavy": 5, "nh": 7,
         "precision": "fp64", "device": True, "rank": 0, "nranks": 1},
        # densities over spherical d shells, the rigorous route
        {"name": "chain7-sph-bound", "kind": "sph", "mol": "chain", "mol_seed": 11, "nheavy": 3, "nh": 4,
         "precision": "bound", "device": True, "rank": 0, "nranks": 1},
        # the Fock-type build of the Lagrangian and the Z-vector equations
        {"name": "chain12-fock", "kind": "fock", "mol": "chain", "mol_seed": 12, "nheavy": 5, "nh": 7,
         "precision": "fp64", "device": False, "rank": 0, "nranks": 1},
        # many small molecules, planned once and replayed
        {"name": "batch3-fp64", "kind": "batch", "mol": "chain", "mol_seed": 40, "nheavy": 1, "nh": 4,
         "precision": "fp64", "device": False, "count": 3, "rank": 0, "nranks": 1},
        # the 32-atom workload, one rank's tiles of a 24-rank run, plain fp64
        {"name": "c2-fp64-1of24", "kind": "grad", "mol": "config", "mol_seed": 1, "nheavy": 13, "nh": 19,
         "precision": "fp64", "device": True, "rank": 0, "nranks": 24},
        # the 32-atom workload on the learned route, one rank's tiles of an 8-rank run
        {"name": "c2-learned-1of8", "kind": "grad", "mol": "config", "mol_seed": 1, "nheavy": 13, "nh": 19,
         "precision": "learned", "device": True, "rank": 0, "nranks": 8},
        # the 300-atom workload: the plan covers the whole system, the kernels one rank's tiles
        {"name": "c4-learned-1of2048", "kind": "grad", "mol": "config", "mol_seed": 3, "nheavy": 129, "nh": 171,
         "precision": "learned", "device": True, "rank": 0, "nranks": 2048},
    ]


def draw(rng):
    kind = rng.choice(["grad", "grad", "grad", "grad", "sph", "fock", "batch"])
    # 1 to 13 heavy atoms (spread over the logarithm) with up to about 1.5 H each
    nheavy = max(1, min(13, int(round(14.0 ** rng.random()))))
    nh = rng.randint(nheavy // 2, nheavy + max(2, nheavy // 2))
    case = {"kind": kind, "mol": "chain", "mol_seed": rng.randint(100, 999), "nheavy": nheavy, "nh": nh,
            "precision": rng.choice(["fp64", "fp64", "bound", "learned"]), "device": rng.random() < 0.5,
            "rank": 0, "nranks": 1}
    if kind == "fock":
        case["precision"], case["device"] = "fp64", False
    if kind in ("fock", "batch"):  # not sharded: the system is kept small
        case["nheavy"], case["nh"] = min(nheavy, 3), min(nh, 5)
        if kind == "batch":
            case["device"], case["count"] = False, rng.randint(2, 5)
            case["precision"] = rng.choice(["fp64", "bound"])
            case["nheavy"] = min(nheavy, 2)
    # a rank of a multi-rank run where the whole gradient takes more than about a second
    est = _estimate(case)
    if kind in ("fock", "batch"):
        while est > 2.5e7 and case["nheavy"] + case["nh"] > 2:
            if case["nh"] > 1:
                case["nh"] -= 1
            else:
                case["nheavy"] -= 1
            est = _estimate(case)
    else:
        case["nranks"] = max(1, int(np.ceil(est / 2.5e7)))
        case["rank"] = rng.randrange(case["nranks"])
    return case


@functools.lru_cache(maxsize=None)
def _skeleton(mol, mol_seed, nheavy, nh):
    """Elements, geometry, basis set and pair coefficients of a molecule."""
    return synth.config(mol_seed) if mol == "config" else synth.molecule(mol_seed, nheavy, nh)


def _estimate(case):
    """Unscreened canonical primitive quartets (one molecule of a batch times the count)."""
    k = _skeleton(case["mol"], case["mol_seed"], case["nheavy"], case["nh"])["shell_nprim"].astype(np.float64)
    n = (k.sum() ** 2 + (k * k).sum()) / 2.0
    return n * n / 2.0 * case.get("count", 1)


def _system(case, seed, shift=0):
    sk = _skeleton(case["mol"], case["mol_seed"] + shift, case["nheavy"], case["nh"])
    rng = np.random.default_rng([seed, shift])
    s = dict(sk)
    s["xyz"] = sk["xyz"] + rng.normal(0.0, 0.02, size=sk["xyz"].shape)
    n = sk["nbf"]
    if case["kind"] == "sph":
        n = int(np.sum(2 * np.asarray(sk["shell_l"]) + 1))

    def density():
        c = rng.normal(0.0, 0.3, size=(n, 5))
        return np.ascontiguousarray(c @ c.T)
    x = rng.normal(size=(n, n))
    x /= np.linalg.norm(x)
    p = density()
    mats = [(p, p), (x, x)] if len(sk["pairs"]) == 2 else [(p, p), (density(), p), (x, x)]
    s["pairs"] = [(a, b) + tuple(old[2:]) for (a, b), old in zip(mats, sk["pairs"])]
    return s


def _router(case):
    return tg.Router(path=ROUTER) if case["precision"] == "learned" else None


def prepare(case, seed):
    router = _router(case)
    if case["kind"] == "batch":
        systems = [_system(case, seed, i) for i in range(case["count"])]
        return {"case": case, "batch": tg.Batch(systems, precision=PRECISION[case["precision"]], router=router),
                "router": router}
    s = _system(case, seed)
    pairs = s["pairs"]
    if case["kind"] == "fock":
        pairs = _fock_pairs(s)
    elif case["device"]:
        put = {}  # a matrix that several pairs share is one tensor
        for a, b, *_ in pairs:
            for m in (a, b):
                put.setdefault(id(m), torch.from_numpy(m).cuda())
        pairs = [(put[id(a)], put[id(b)], *rest) for a, b, *rest in pairs]
    return {"case": case, "basis": tg.Basis(s), "pairs": pairs, "router": router}


def _fock_pairs(s):
    """The Lagrangian's Fock-type matrix over the difference density plus the
    Z-vector's over the transition density."""
    return [(np.ascontiguousarray(s["pairs"][1][0].T), 2.0, -0.157706, -0.842294, 0.3)] + \
        tg.zfock_pairs(s["pairs"][-1][0], 0.157706, 0.842294, 0.3)


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        return state["batch"].run()[0]
    if case["kind"] == "fock":
        return state["basis"].fock2e(state["pairs"], screen_tol=1e-10)[0]
    g, _ = state["basis"].grad2e(state["pairs"], precision=PRECISION[case["precision"]], router=state["router"],
                                 rank=case["rank"], nranks=case["nranks"],
                                 shard_mode=tg.TG_SHARD_TILES if case["nranks"] > 1 else tg.TG_SHARD_PAIR_KEY,
                                 spherical=case["kind"] == "sph")
    return g


def work(case):
    """Bytes: every density matrix and basis record read once, the result
    written once.  Flops of a primitive quartet and operator, whatever the
    algorithm: the Boys orders and the Hermite Coulomb tensor they start (one
    multiply-add per entry of every level), one multiply-add per pair of bra
    and ket Hermite indices, and the four sums of the energy and its three
    shift derivatives.  The primitive quartets are counted by the library."""
    state = prepare(case, 0)
    fock = case["kind"] == "fock"
    if case["kind"] == "batch":
        st = state["batch"].run()[1]
        nat = sum(state["batch"].natoms)
        size = sum(2 * m.nbytes for keep in state["batch"]._keep for m in keep[:1]) * 3 // 2
        out = nat * 24
    else:
        if fock:
            st = state["basis"].fock2e(state["pairs"], screen_tol=1e-10)[1]
        else:
            st = state["basis"].grad2e(state["pairs"], precision=PRECISION[case["precision"]], router=state["router"],
                                       rank=case["rank"], nranks=case["nranks"],
                                       shard_mode=1 if case["nranks"] > 1 else 0, spherical=case["kind"] == "sph")[1]
        mats = {}
        for t in state["pairs"]:
            for m in t[:1] if fock else t[:2]:
                mats[id(m)] = m.nbytes
        size = sum(mats.values())
        out = state["basis"].nbf ** 2 * 8 if fock else state["basis"].natom * 24
    nherm = lambda n: (n + 1) * (n + 2) * (n + 3) // 6  # noqa: E731
    flops = 0.0
    for qc in range(21):
        P = max(i for i in range(6) if i * (i + 1) // 2 <= qc)
        l1, l2 = ((0, 1, 2, 2, 3, 4)[i] for i in (P, qc - P * (P + 1) // 2))
        top = l1 + l2 + (0 if fock else 1)
        levels = sum(nherm(k) - 1 for k in range(1, top + 1))
        per = 2 * (6 + 2 * top) + 2 * levels + 2 * nherm(l1) * nherm(l2) + (0 if fock else 8 * nherm(l1 + l2))
        n = st["class_prim_quartets"][qc] + (0 if fock else st["class_prim_quartets_fp32"][qc])
        flops += 2.0 * per * n
    return {"bytes": float(size + out), "flops": flops}


# ---------------------------------------------------------------- plain 64-bit evaluation
#
# The energy E = sum_pairs sum [c_J (mn|ls) A_mn B_ls + c_K (mn|ls) A_ml B_ns + lr] over all
# canonical shell quartets, written with the McMurchie-Davidson expansion in torch and
# differentiated by autograd: with respect to the nuclei for the gradient, with respect to A
# for the Fock-type matrix.  No screening.


class _Boys(torch.autograd.Function):
    @staticmethod
    def forward(ctx, T, M):
        F = [None] * (M + 2)
        small = T < 30.0
        Ts = torch.where(small, T, torch.ones_like(T))
        term = torch.full_like(Ts, 1.0 / (2 * M + 3))
        acc = term.clone()
        for k in range(1, 140):
            term = term * (2.0 * Ts / (2 * M + 3 + 2 * k))
            acc += term
        e = torch.exp(-Ts)
        F[M + 1] = e * acc
        for m in range(M, -1, -1):
            F[m] = (2.0 * Ts * F[m + 1] + e) / (2 * m + 1)
        Tl = torch.where(small, torch.full_like(T, 30.0), T)
        el = torch.exp(-Tl)
        f = 0.5 * torch.sqrt(np.pi / Tl) * torch.erf(torch.sqrt(Tl))
        for m in range(M + 2):
            F[m] = torch.where(small, F[m], f)
            f = ((2 * m + 1) * f - el) / (2.0 * Tl)
        F = torch.stack(F)
        ctx.save_for_backward(F)
        return F[:-1].clone()

    @staticmethod
    def backward(ctx, g):
        F, = ctx.saved_tensors
        return -(g * F[1:]).sum(0), None


def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _herm(L):
    return [(t, u, n - t - u) for n in range(L + 1) for t in range(n, -1, -1) for u in range(n - t, -1, -1)]


def _expansion(la, lb, PA, PB, oo2p):
    """E[ab, h, N] of every component pair from 1-D recursions (PA, PB: [3, N])."""
    one, zero = torch.ones_like(PA), torch.zeros_like(PA)
    E = {(0, 0): [one]}

    def at(e, t):
        return e[t] if 0 <= t < len(e) else zero

    def up(e, X):
        return [X * at(e, t) + oo2p * at(e, t - 1) + (t + 1) * at(e, t + 1) for t in range(len(e) + 1)]
    for i in range(la + 1):
        if i:
            E[i, 0] = up(E[i - 1, 0], PA)
        for j in range(1, lb + 1):
            E[i, j] = up(E[i, j - 1], PB)
    hs = _herm(la + lb)
    rows = []
    for a in _cart(la):
        for b in _cart(lb):
            rows.append(torch.stack([at(E[a[0], b[0]], h[0])[0] * at(E[a[1], b[1]], h[1])[1] *
                                     at(E[a[2], b[2]], h[2])[2] for h in hs]))
    return torch.stack(rows)


def _hermite_R(L, base, X):
    R = {(L, (0, 0, 0)): base[L]}
    for n in range(L - 1, -1, -1):
        R[n, (0, 0, 0)] = base[n]
        for h in _herm(L - n)[1:]:
            d = next(i for i in range(3) if h[i])
            h1 = tuple(h[i] - (i == d) for i in range(3))
            v = X[d] * R[n + 1, h1]
            if h[d] > 1:
                v = v + (h[d] - 1) * R[n + 1, tuple(h[i] - 2 * (i == d) for i in range(3))]
            R[n, h] = v
    return torch.stack([R[0, h] for h in _herm(L)])


def _differentiate(s, pairs, wrt):
    """dE/d(xyz) (wrt "xyz") or dE/dA of the pairs' first matrices (wrt "A") as a numpy array."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f8 = dict(dtype=torch.float64, device=dev)
    xyz = torch.tensor(s["xyz"] - s["xyz"].mean(0), **f8)
    nbf = pairs[0][0].shape[0]
    mats = [(torch.tensor(a, **f8), torch.tensor(b, **f8)) for a, b, *_ in pairs]
    leaf = xyz.requires_grad_() if wrt == "xyz" else torch.zeros((nbf, nbf), requires_grad=True, **f8)
    if wrt == "A":
        mats = [(leaf, b) for _, b in mats]
    l, npr, at = np.asarray(s["shell_l"]), np.asarray(s["shell_nprim"]), np.asarray(s["shell_atom"])
    bf = np.concatenate([[0], np.cumsum([(k + 1) * (k + 2) // 2 for k in l])])
    off = np.concatenate([[0], np.cumsum(npr)])
    lp = np.repeat(l, npr)
    ex, fact2 = s["exps"], np.array([1.0, 1.0, 3.0])
    co = s["coefs"] * (2 * ex / np.pi) ** 0.75 * (4 * ex) ** (lp / 2.0) / np.sqrt(fact2[lp])
    for i in range(len(l)):  # contracted norm of the x^l component
        sl = slice(off[i], off[i + 1])
        z = ex[sl][:, None] + ex[sl][None]
        S = (np.pi / z) ** 1.5 * fact2[l[i]] / (2 * z) ** l[i]
        co[sl] /= np.sqrt(co[sl] @ S @ co[sl])
    omega = max([p[5] for p in pairs if p[4] != 0.0] + [0.0])
    shells = {k: [] for k in range(6)}
    for i in range(len(l)):
        for j in range(i + 1):
            a, b = (i, j) if l[i] >= l[j] else (j, i)
            shells[l[a] * (l[a] + 1) // 2 + l[b]].append((a, b))
    ten = lambda v, **k: torch.tensor(np.ascontiguousarray(v), device=dev, **k)  # noqa: E731
    for P in range(6):
        for Q in range(P + 1):
            bra, ket = np.array(shells[P]).reshape(-1, 2), np.array(shells[Q]).reshape(-1, 2)
            if not len(bra) or not len(ket):
                continue
            I, J = np.meshgrid(np.arange(len(bra)), np.arange(len(ket)), indexing="ij")
            keep = (I >= J) if P == Q else np.ones_like(I, bool)
            quart = np.concatenate([bra[I[keep]], ket[J[keep]]], axis=1)
            nq = npr[quart].prod(1)
            (la, lb), (lc, ld) = [tuple(int(l[k]) for k in x[0]) for x in (bra, ket)]
            nf = [(k + 1) * (k + 2) // 2 for k in (la, lb, lc, ld)]
            cap = max(2000, 60_000_000 // (nf[0] * nf[1] * nf[2] * nf[3] + 12 * len(_herm(la + lb + lc + ld + 1)) * 4))
            order, at0 = np.argsort(nq, kind="stable"), 0
            while at0 < len(order):
                cum = np.cumsum(nq[order[at0:at0 + cap]])
                take = max(1, int(np.searchsorted(cum, cap, side="right")))
                _energy(quart[order[at0:at0 + take]], (la, lb, lc, ld), nf, xyz, mats, pairs, omega, at, bf, off, npr,
                        ex, co, ten).backward()
                at0 += take
    return leaf.grad.cpu().numpy()


def _energy(quart, ls, nf, xyz, mats, pairs, omega, at, bf, off, npr, ex, co, ten):
    a, b, c, d = quart.T
    scale = np.where(a == b, 0.5, 1.0) * np.where(c == d, 0.5, 1.0) * np.where((a == c) & (b == d), 0.5, 1.0)
    ix = [ten(bf[x][:, None] + np.arange(n)[None]) for x, n in zip((a, b, c, d), nf)]
    m, n, p, q = (ix[0][:, :, None, None, None], ix[1][:, None, :, None, None], ix[2][:, None, None, :, None],
                  ix[3][:, None, None, None, :])
    gam = [0.0, 0.0]
    for (A, B), (_, _, cj, ck, cl, _om) in zip(mats, pairs):
        if cj:
            S, T = A + A.T, B + B.T
            gam[0] = gam[0] + cj * (S[m, n] * T[p, q] + S[p, q] * T[m, n])
        if ck or (cl and omega > 0):
            k = 0.0
            for u, v in ((m, n), (n, m)):
                for w, z in ((p, q), (q, p)):
                    k = k + A[u, w] * B[v, z] + A[w, u] * B[z, v]
            gam[0] = gam[0] + ck * k
            if cl and omega > 0:
                gam[1] = gam[1] + cl * k
    # primitive quartets of every contracted one
    cnt = npr[quart].prod(1)
    own = np.repeat(np.arange(len(quart)), cnt)
    r = np.arange(len(own)) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    pr = [None] * 4
    for k in (3, 2, 1, 0):
        pr[k] = off[quart[own, k]] + r % npr[quart[own, k]]
        r = r // npr[quart[own, k]]
    za, zb, zc, zd = (ten(ex[k]) for k in pr)
    A, B, C, D = (xyz[ten(at[quart[own, k]])].T for k in range(4))
    pz, qz = za + zb, zc + zd
    AB, CD = A - B, C - D
    K = ten(co[pr[0]] * co[pr[1]] * co[pr[2]] * co[pr[3]] * scale[own]) * \
        torch.exp(-za * zb / pz * (AB * AB).sum(0) - zc * zd / qz * (CD * CD).sum(0))
    Eb = _expansion(ls[0], ls[1], -(zb / pz) * AB, (za / pz) * AB, 0.5 / pz)
    Ek = _expansion(ls[2], ls[3], -(zd / qz) * CD, (zc / qz) * CD, 0.5 / qz)
    X = (A - C) - (zb / pz) * AB + (zd / qz) * CD
    rho = pz * qz / (pz + qz)
    T = rho * (X * X).sum(0)
    pref = 2 * np.pi ** 2.5 / (pz * qz * torch.sqrt(pz + qz)) * K
    L = sum(ls)
    h1, h2 = _herm(ls[0] + ls[1]), _herm(ls[2] + ls[3])
    pos = {h: i for i, h in enumerate(_herm(L))}
    at_r = torch.tensor([[pos[tuple(u + v for u, v in zip(x, y))] for y in h2] for x in h1], device=T.device)
    sign = torch.tensor([(-1.0) ** sum(y) for y in h2], dtype=T.dtype, device=T.device)
    own_t = ten(own)
    total = 0.0
    for op, g in enumerate(gam):
        if isinstance(g, float):
            continue
        th2 = torch.ones_like(rho) if op == 0 else omega * omega / (omega * omega + rho)
        F = _Boys.apply(T * th2, L)
        R = _hermite_R(L, [pref * torch.sqrt(th2) * (-2.0 * rho * th2) ** n * F[n] for n in range(L + 1)], X)
        RR = R[at_r.reshape(-1)].reshape(len(h1), len(h2), -1) * sign[None, :, None]
        G = g.reshape(len(quart), nf[0] * nf[1], nf[2] * nf[3])[own_t]                     # N, ab, cd
        W = torch.bmm(Eb.permute(2, 0, 1), RR.permute(2, 0, 1))                             # N, ab, h2
        total = total + (torch.bmm(W, Ek.permute(2, 1, 0)) * G).sum()
    return total


def _to_cartesian(s):
    """The nbf x nsph matrix of the spherical functions (d: xy, yz, z2, xz, x2-y2 of unit norm)."""
    r3 = np.sqrt(3.0)
    d = np.zeros((6, 5))
    d[1, 0], d[4, 1], d[2, 3] = r3, r3, r3
    d[5, 2], d[0, 2], d[3, 2] = 1.0, -0.5, -0.5
    d[0, 4], d[3, 4] = 0.5 * r3, -0.5 * r3
    blocks = [d if k == 2 else np.eye(2 * k + 1) for k in s["shell_l"]]
    T = np.zeros((sum(x.shape[0] for x in blocks), sum(x.shape[1] for x in blocks)))
    i = j = 0
    for x in blocks:
        T[i:i + x.shape[0], j:j + x.shape[1]] = x
        i, j = i + x.shape[0], j + x.shape[1]
    return T


def exact(case, seed):
    if case["nranks"] > 1 or _estimate(case) > 2e7:
        return None
    if case["kind"] == "batch":
        return [_differentiate(s, s["pairs"], "xyz") for s in (_system(case, seed, i) for i in range(case["count"]))]
    s = _system(case, seed)
    if case["kind"] == "fock":
        return _differentiate(s, [(b, b, *rest) for b, *rest in _fock_pairs(s)], "A")
    pairs = s["pairs"]
    if case["kind"] == "sph":
        T = _to_cartesian(s)
        pairs = [(T @ a @ T.T, T @ b @ T.T, *rest) for a, b, *rest in pairs]
    return _differentiate(s, pairs, "xyz")
