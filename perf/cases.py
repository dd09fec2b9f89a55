"""The work that a user of the engine has it do, as cases that can be timed and compared.

`listed()` gives the cases, `draw(rng)` more of the same ranges, `prepare` what a program holds before the call (basis
on the device, index lists, prepared batches, densities, Schwarz factors), `run` one pass through the public entry
points, `work` the bytes and operations of one pass, and `exact` the same results from plain torch operations in
64 bits (dense McMurchie-Davidson matrices, autograd for the gradient), written without the engine.
"""
import functools
import math

import numpy as np
import torch

from paper_2405_01834_gb300 import inputs, mdx

MAX_OUT = 300_000_000          # doubles of one pass's output (the largest listed case writes 280 M)
MAX_FLOPS = 45e9               # operations of one drawn class-grid pass (the largest listed grid does 11e9; see work)
EXACT_FLOPS = 2.5e12           # dense operations above which exact() would take too long
_ENGINE = None


def engine():
    """One engine for the process, as a program keeps it: it holds the tables, class plans and workspace."""
    global _ENGINE
    if _ENGINE is None:
        _ENGINE = mdx.Engine(0)
    return _ENGINE


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # The integrals of a water-sized molecule in one call: a few hundred quartets over 36 classes, so launches and
        # the host's preparation of the call count.
        {"name": "eri4_call_2atoms", "kind": "eri4", "atoms": 2, "lmax": 2, "K": 3, "every": 1},
        # All 14,706 unique quartets of the repository's first configuration (6 atoms, s/p/d, K = 3) in one call.
        {"name": "eri4_call_6atoms", "kind": "eri4", "atoms": 6, "lmax": 2, "K": 3, "every": 1},
        # The benchmark's class sweep (prepared batches): the smallest class at its full 224 x 224 grid, ...
        {"name": "batch_pppp", "kind": "grid4", "l": "1111", "K": "1111", "nb": 224, "nk": 224, "sph": False},
        # ... an odd-sized grid of the polarisation class [dd|dd], ...
        {"name": "batch_dddd", "kind": "grid4", "l": "2222", "K": "1111", "nb": 181, "nk": 173, "sph": False},
        # ... [ff|ff], the middle of the sweep, ...
        {"name": "batch_ffff", "kind": "grid4", "l": "3333", "K": "1111", "nb": 96, "nk": 75, "sph": False},
        # ... and one 456-quartet chunk of its largest class, [ii|ii] (2.2 GB of integrals).
        {"name": "batch_iiii", "kind": "grid4", "l": "6666", "K": "1111", "nb": 24, "nk": 19, "sph": False},
        # A mixed contracted class as the s (K = 6), p (K = 3) and d (K = 1) shells of the molecular basis make it.
        {"name": "batch_dpps_contracted", "kind": "grid4", "l": "2110", "K": "1336", "nb": 201, "nk": 167, "sph": False},
        # Solid-harmonic output (the basis of production calculations), [33|33] with a contracted ket.
        {"name": "sph_ffff_contracted", "kind": "grid4", "l": "3333", "K": "1115", "nb": 61, "nk": 50, "sph": True},
        # Density fitting: every [a|cd] of a 4-atom cluster, s..i auxiliary shells on a 4s3p2d1f orbital basis.
        {"name": "df_4atoms", "kind": "df", "atoms": 4, "every": 1},
        # One exchange build of an SCF iteration: 5-atom cluster in the 5s4p3d2f1g / 4s3p2d1f basis.
        {"name": "exchange_5atoms", "kind": "exchange", "heavy": 2, "light": 3, "tau": 1e-11},
        # The exchange part of one geometry step: energy and nuclear gradient of a 3-atom molecule.
        {"name": "gradient_3atoms", "kind": "gradient", "heavy": 1, "light": 2, "tau": 1e-11},
        # A data-generation batch: the exchange matrices of 8 small molecules of uneven size (1 to 3 atoms), one
        # prepared batch, launched per class.
        {"name": "xbatch_8mol", "kind": "xbatch", "molecules": 8, "lo": 1, "hi": 3, "tau": 1e-11, "mode": 0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["eri4", "grid4", "grid4", "grid4", "sph4", "df", "exchange", "gradient", "xbatch"])
    if kind == "eri4":
        lmax = rng.choice([1, 2, 2, 3])
        return {"kind": "eri4", "atoms": rng.randint(1, 3 if lmax == 3 else 6), "lmax": lmax, "K": rng.randint(1, 4),
                "every": rng.choice([1, 1, 2, 5])}
    if kind in ("grid4", "sph4"):
        while True:
            l = [rng.randint(0, 6) for _ in range(4)] if rng.random() < 0.5 else [rng.randint(0, 6)] * 4
            K = [rng.choice([1, 1, 2, 3, 6]) if x < 2 else rng.choice([1, 1, 1, 2]) for x in l]
            c = {"kind": "grid4", "l": "".join(map(str, l)), "K": "".join(map(str, K)), "nb": 1, "nk": 1,
                 "sph": kind == "sph4"}
            one = work(c)
            cap = int(min(60000, MAX_OUT / _grid_out(c), MAX_FLOPS / 4 / one["flops"],
                          3e11 / _dense_flops(l, K)))
            if cap < 4:
                continue
            n = _log_int(rng, min(64, cap), cap)
            c["nb"] = _log_int(rng, max(1, int(math.sqrt(n) / 3)), max(1, int(math.sqrt(n))))
            c["nk"] = max(1, n // c["nb"])
            return c
    if kind == "df":
        return {"kind": "df", "atoms": rng.randint(1, 4), "every": rng.randint(1, 16)}
    tau = rng.choice([1e-9, 1e-10, 1e-11, 1e-12, 0.0])
    if kind in ("exchange", "gradient"):   # at least two atoms: the gradient of one is zero
        heavy = rng.randint(0, 2)
        light = rng.randint(max(0, 2 - heavy), (5 if kind == "exchange" else 3) - heavy)
        return {"kind": kind, "heavy": heavy, "light": light, "tau": tau}
    lo = rng.randint(1, 2)
    return {"kind": "xbatch", "molecules": rng.randint(2, 8), "lo": lo, "hi": rng.randint(lo, 3), "tau": tau,
            "mode": rng.choice([0, 1, 2])}


# ------------------------------------------------------------------------------------------------ inputs
def _digits(text):
    return tuple(int(c) for c in text)


def _grid_out(case):
    l = _digits(case["l"])
    n = [2 * x + 1 if case["sph"] else inputs.ncart(x) for x in l]
    return n[0] * n[1] * n[2] * n[3]


def _triplets(case, aux, orb):
    cd = [(c, d) for c in range(orb.n_shells) for d in range(c + 1)]
    t = np.array([(a, c, d) for a in range(aux.n_shells) for c, d in cd], dtype=np.int32)
    return t[:: case["every"]]


def _pairs(n):
    return np.array([(i, j) for i in range(n) for j in range(i + 1)], dtype=np.int32)


def _molecule(seed, heavy, light):
    """A compact cluster of `heavy` 5s4p3d2f1g and `light` 4s3p2d1f atoms (the recipe of inputs.molecule with the
    number of each fixed, so that the seed does not change the size of the matrices)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    xyz = inputs.cluster(rng, heavy + light)
    bb = inputs.BasisBuilder()
    for a, x in enumerate(xyz):
        bb.add_atom(x)
        for l, n, K in inputs.HEAVY_SHELLS if a < heavy else inputs.LIGHT_SHELLS:
            for i in range(n):
                z = 0.1 * 2.0 ** l * 2.5 ** i * 3.5 ** np.arange(K)
                c = rng.uniform(0.1, 1.0, K) * inputs.primitive_norm(l, z)
                bb.add_shell(l, x, z, c / math.sqrt(inputs.contracted_self_overlap(l, z, c)), a)
    return bb.build()


def _host_inputs(case, seed):
    """The bases, index lists and densities of a case, on the host."""
    kind = case["kind"]
    if kind == "eri4":
        b = inputs.small_molecule(seed=1001 + seed, n_atoms=case["atoms"], K=case["K"], shells=tuple(range(case["lmax"] + 1)))
        return {"basis": b, "quartets": inputs.unique_quartets(b.n_shells)[:: case["every"]]}
    if kind == "grid4":
        b, q = inputs.class_sweep(_digits(case["l"]), case["nb"], case["nk"], seed=1002 + seed, K=_digits(case["K"]))
        return {"basis": b, "quartets": q}
    if kind == "df":
        aux, orb = inputs.df_cluster(seed=1003 + seed, n_atoms=case["atoms"])
        return {"aux": aux, "orb": orb, "triplets": _triplets(case, aux, orb)}
    if kind in ("exchange", "gradient"):
        b = _molecule(1005 + seed, case["heavy"], case["light"])
        return {"basis": b, "D": inputs.density(b.nao, 11 + seed)}
    sizes = [case["lo"] + i % (case["hi"] - case["lo"] + 1) for i in range(case["molecules"])]
    mols = [_molecule(1004000 + 64 * seed + i, (n + i % 2) // 2, n - (n + i % 2) // 2) for i, n in enumerate(sizes)]
    return {"bases": mols, "Ds": [inputs.density(b.nao, 17 + seed + i) for i, b in enumerate(mols)]}


def prepare(case, seed):
    """What the program has in hand: device bases and index lists, a prepared batch and its output buffer, pairs with
    their Schwarz factors and a density."""
    eng, h, kind = engine(), _host_inputs(case, seed), case["kind"]
    gpu = lambda a, dt: torch.as_tensor(a, dtype=dt, device="cuda")  # noqa: E731
    s = {"kind": kind, "eng": eng}
    if kind == "eri4":
        s["basis"], s["quartets"] = mdx.DeviceBasis(h["basis"]), gpu(h["quartets"], torch.int32)
    elif kind == "grid4":
        s["basis"] = mdx.DeviceBasis(h["basis"])
        make = eng.batch_eri4_sph if case["sph"] else eng.batch_eri4
        s["batch"] = make(s["basis"], gpu(h["quartets"], torch.int32))
        s["out"] = torch.empty(s["batch"].total, dtype=torch.float64, device="cuda")
    elif kind == "df":
        s["aux"], s["orb"] = mdx.DeviceBasis(h["aux"]), mdx.DeviceBasis(h["orb"])
        s["batch"] = eng.batch_eri3(s["aux"], s["orb"], gpu(h["triplets"], torch.int32))
        s["out"] = torch.empty(s["batch"].total, dtype=torch.float64, device="cuda")
    elif kind in ("exchange", "gradient"):
        s["basis"], s["D"] = mdx.DeviceBasis(h["basis"]), gpu(h["D"], torch.float64)
        s["pairs"] = gpu(_pairs(h["basis"].n_shells), torch.int32)
        s["Q"], s["tau"] = eng.schwarz(s["basis"], s["pairs"]), case["tau"]
    else:
        s["xb"] = eng.xbatch([mdx.DeviceBasis(b) for b in h["bases"]], [gpu(d, torch.float64) for d in h["Ds"]], tau=case["tau"])
        s["mode"] = case["mode"]
    return s


def run(state):
    eng, kind = state["eng"], state["kind"]
    if kind == "eri4":
        return eng.eri4(state["basis"], state["quartets"])
    if kind in ("grid4", "df"):
        state["batch"].run(state["out"])
        return state["out"]
    if kind == "exchange":
        return eng.exchange(state["basis"], state["pairs"], state["Q"], state["D"], tau=state["tau"], alpha=-1.0)
    if kind == "gradient":
        return eng.exchange_grad(state["basis"], state["pairs"], state["Q"], state["D"], tau=state["tau"])
    state["xb"].run(state["mode"])
    return state["xb"].Ks


# ------------------------------------------------------------------------------------------------ work
def _class_flops(l, K, count=1.0, n_out=None):
    """Operations that a class of shellsets cannot do without: per primitive quartet its nherm(L) Hermite integrals (an
    FMA each); per output element a product of three axes at floor(L/2) + 1 quadrature points (a multiply and an FMA
    each), the fewest of the known forms that keep full accuracy, for one primitive quartet."""
    L = sum(l)
    if n_out is None:
        n_out = math.prod(inputs.ncart(x) for x in l)
    return count * (2.0 * math.prod(K) * (L + 1) * (L + 2) * (L + 3) / 6 + 3.0 * (L // 2 + 1) * n_out)


def _count_classes(l, K, pairs):
    """{(l, K of a pair): number of pairs}."""
    found = {}
    for i, j in pairs:
        key = (int(l[i]), int(l[j]), int(K[i]), int(K[j]))
        found[key] = found.get(key, 0) + 1
    return found


def _exchange_flops(basis):
    """All unique quartets of the shell pairs (screening drops few of these compact molecules)."""
    cls = sorted(_count_classes(basis.l, basis.nprim, _pairs(basis.n_shells)).items())
    tot = 0.0
    for x, (p, n) in enumerate(cls):
        for q, m in cls[: x + 1]:
            tot += _class_flops((p[0], p[1], q[0], q[1]), (p[2], p[3], q[2], q[3]), n * (n + 1) / 2 if p == q else n * m)
    return tot


def work(case):
    kind = case["kind"]
    if kind == "grid4":
        n = case["nb"] * case["nk"]
        one = _grid_out(case)
        return {"bytes": 8.0 * n * one + 16.0 * n, "flops": _class_flops(_digits(case["l"]), _digits(case["K"]), n, one)}
    h = _host_inputs(case, 1)
    if kind == "eri4":
        b, q = h["basis"], h["quartets"]
        l, K = b.l[q], b.nprim[q]
        flops = n_out = 0.0
        for key, n in zip(*np.unique(np.concatenate([l, K], axis=1), axis=0, return_counts=True)):
            flops += _class_flops([int(x) for x in key[:4]], [int(x) for x in key[4:]], int(n))
            n_out += int(n) * math.prod(inputs.ncart(int(x)) for x in key[:4])
        return {"bytes": 8.0 * n_out + 24.0 * len(q), "flops": flops}
    if kind == "df":
        aux, orb, t = h["aux"], h["orb"], h["triplets"]
        keys = np.stack([aux.l[t[:, 0]], orb.l[t[:, 1]], orb.l[t[:, 2]], aux.nprim[t[:, 0]], orb.nprim[t[:, 1]],
                         orb.nprim[t[:, 2]]], axis=1)
        flops = n_out = 0.0
        for key, n in zip(*np.unique(keys, axis=0, return_counts=True)):
            flops += _class_flops([int(x) for x in key[:3]], [int(x) for x in key[3:]], int(n))
            n_out += int(n) * math.prod(inputs.ncart(int(x)) for x in key[:3])
        return {"bytes": 8.0 * n_out + 12.0 * len(t), "flops": flops}
    if kind == "exchange":
        return {"bytes": 16.0 * h["basis"].nao ** 2, "flops": _exchange_flops(h["basis"])}
    if kind == "gradient":   # the integrals once, and their three axes' derivatives
        return {"bytes": 8.0 * h["basis"].nao ** 2 + 24.0 * h["basis"].n_atoms, "flops": 2.5 * _exchange_flops(h["basis"])}
    return {"bytes": sum(16.0 * b.nao ** 2 for b in h["bases"]), "flops": sum(_exchange_flops(b) for b in h["bases"])}


# ------------------------------------------------------------------------------------------------ 64-bit results
def _dense_flops(l, K):
    """Operations of the dense matrix form of one shellset (the form exact() uses)."""
    nh = lambda n: (n + 1) * (n + 2) * (n + 3) / 6  # noqa: E731
    hb, hk = nh(l[0] + l[1]), nh(l[2] + l[3])
    nb, nk = inputs.ncart(l[0]) * inputs.ncart(l[1]), inputs.ncart(l[2]) * inputs.ncart(l[3])
    return 2 * K[0] * K[1] * hb * nk * (K[2] * K[3] * hk + nb) + 40 * math.prod(K) * (nh(sum(l)) + 60)


def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


@functools.lru_cache(maxsize=None)
def _hermite(n):
    return [(t, u, v) for t in range(n + 1) for u in range(n + 1 - t) for v in range(n + 1 - t - u)]


class _Boys(torch.autograd.Function):
    """F_m(T), m = 0..n: the ascending series at m = n and downward recursion, or erf and upward recursion (T > 40)."""

    @staticmethod
    def forward(ctx, T, n):
        F = torch.empty(T.shape + (n + 2,), dtype=T.dtype, device=T.device)
        small = T.clamp(max=40.0)
        ex = torch.exp(-small)
        term = torch.full_like(T, 1.0 / (2 * n + 3))
        acc = term.clone()
        for i in range(1, 121):
            term = term * (2.0 * small / (2 * n + 3 + 2 * i))
            acc = acc + term
        F[..., n + 1] = ex * acc
        for m in range(n, -1, -1):
            F[..., m] = (2.0 * small * F[..., m + 1] + ex) / (2 * m + 1)
        big = T.clamp(min=40.0)
        ex = torch.exp(-big)
        G = 0.5 * torch.sqrt(math.pi / big) * torch.erf(torch.sqrt(big))
        for m in range(n + 2):
            F[..., m] = torch.where(T > 40.0, G, F[..., m])
            G = ((2 * m + 1) * G - ex) / (2.0 * big)
        ctx.save_for_backward(F)
        return F[..., : n + 1].clone()

    @staticmethod
    def backward(ctx, g):
        (F,) = ctx.saved_tensors
        return -(g * F[..., 1:]).sum(-1), None


@functools.lru_cache(maxsize=None)
def _gather(Lb, Lk):
    """Place of [p + q] in the order-L_b+L_k list, for every pair of Hermite functions p and q."""
    at = {h: i for i, h in enumerate(_hermite(Lb + Lk))}
    return torch.tensor([at[tuple(x + y for x, y in zip(p, q))] for p in _hermite(Lb) for q in _hermite(Lk)], device="cuda")


@functools.lru_cache(maxsize=None)
def _r_levels(L):
    """Index lists of [tuv]^(n) = X [tuv - 1]^(n+1) + k [tuv - 2]^(n+1), by total order."""
    levels = []
    for N in range(1, L + 1):
        at = {h: i for i, h in enumerate(_hermite(N - 1))}
        axis, one, two, k = [], [], [], []
        for h in _hermite(N):
            ax = max((i for i in range(3) if h[i] > 0), default=0)
            lower = lambda n: at.get(tuple(h[i] - (n if i == ax else 0) for i in range(3)), 0)  # noqa: E731
            axis.append(ax)
            one.append(lower(1) if any(h) else 0)
            two.append(lower(2) if h[ax] > 1 else 0)
            k.append(float(h[ax] - 1) if h[ax] > 1 else 0.0)
        levels.append(tuple(torch.tensor(x, device="cuda") for x in (axis, one, two, k)))
    return levels


class _PairSet:
    """Unique shell pairs of one class: exponents, centres and dense Cartesian-to-Hermite matrices per primitive pair."""

    def __init__(self, bas, coords, pairs, sign):
        i, j = pairs[:, 0], pairs[:, 1]
        dev = coords.device
        one = int(j[0]) < 0
        self.la, self.lb = int(bas.l[i[0]]), 0 if one else int(bas.l[j[0]])
        Ka, Kb = int(bas.nprim[i[0]]), 1 if one else int(bas.nprim[j[0]])
        prim = lambda a, s, K: torch.as_tensor(a[bas.prim_off[s][:, None] + np.arange(K)], device=dev)  # noqa: E731
        A = coords[torch.as_tensor(i, dtype=torch.long, device=dev)]
        ea, ca = prim(bas.exps, i, Ka), prim(bas.coefs, i, Ka)
        if one:
            B, eb, cb = A, torch.zeros_like(ea[:, :1]), torch.ones_like(ea[:, :1])
        else:
            B = coords[torch.as_tensor(j, dtype=torch.long, device=dev)]
            eb, cb = prim(bas.exps, j, Kb), prim(bas.coefs, j, Kb)
        self.K, n = Ka * Kb, len(pairs)
        za, zb = ea[:, :, None].expand(n, Ka, Kb).reshape(n, -1), eb[:, None, :].expand(n, Ka, Kb).reshape(n, -1)
        c = (ca[:, :, None] * cb[:, None, :]).reshape(n, -1)
        self.p = za + zb
        self.P = (za[..., None] * A[:, None] + zb[..., None] * B[:, None]) / self.p[..., None]
        c = c * torch.exp(-za * zb / self.p * ((A - B) ** 2).sum(-1)[:, None])
        XA, XB, h = self.P - A[:, None], self.P - B[:, None], (0.5 / self.p)[..., None]
        la, lb, L = self.la, self.lb, self.la + self.lb
        E = {(0, 0): [torch.ones_like(XA)]}

        def up(row, X):
            out = []
            for t in range(len(row) + 1):
                v = h * row[t - 1] if t else 0.0
                if t < len(row):
                    v = v + X * row[t]
                if t + 1 < len(row):
                    v = v + (t + 1) * row[t + 1]
                out.append(v)
            return out

        for a in range(la + 1):
            if a:
                E[a, 0] = up(E[a - 1, 0], XA)
            for b in range(lb):
                E[a, b + 1] = up(E[a, b], XB)
        zero = torch.zeros_like(XA)
        tab = torch.stack([torch.stack([torch.stack(E[a, b] + [zero] * (L - a - b), -1) for b in range(lb + 1)], -2)
                           for a in range(la + 1)], -3)                                  # [n, K, 3, la+1, lb+1, L+1]
        herm = _hermite(L)
        ab = [(x, y) for x in _cart(la) for y in _cart(lb)]
        M = c[..., None, None]
        for ax in range(3):
            row = tab[:, :, ax, [x[ax] for x, _ in ab], [y[ax] for _, y in ab]]          # [n, K, N, L+1]
            M = M * row[..., [t[ax] for t in herm]]
        if sign:
            M = M * torch.tensor([(-1.0) ** sum(t) for t in herm], dtype=M.dtype, device=dev)
        self.M = M                                                                       # [n, K, N, H]


def _blocks(bb, cb, bk, ck, bra, ket, limit=1.2e9):
    """Integrals of the quartets (bra[q] | ket[q]) by class: yields (quartet numbers, [n, N_bra, N_ket]). Pairs with a
    second index -1 have one centre. `cb`, `ck`: shell centres (tensors) of the two bases."""
    dev = cb.device

    def key_of(bas, pr):
        j, one = np.maximum(pr[:, 1], 0), pr[:, 1] < 0
        return np.stack([bas.l[pr[:, 0]], np.where(one, 0, bas.l[j]), bas.nprim[pr[:, 0]], np.where(one, 1, bas.nprim[j])], 1)

    keys = np.concatenate([key_of(bb, bra), key_of(bk, ket)], axis=1)
    _, inv = np.unique(keys, axis=0, return_inverse=True)
    inv = inv.reshape(-1)
    order = np.argsort(inv, kind="stable")
    for idx in np.split(order, np.flatnonzero(np.diff(inv[order])) + 1):
        k = [int(x) for x in keys[idx[0]]]
        L, Lb, Lk = k[0] + k[1] + k[4] + k[5], k[0] + k[1], k[4] + k[5]
        Kb, Kk, hb, hk = k[2] * k[3], k[6] * k[7], len(_hermite(Lb)), len(_hermite(Lk))
        nb, nk = inputs.ncart(k[0]) * inputs.ncart(k[1]), inputs.ncart(k[4]) * inputs.ncart(k[5])
        ub, ib = np.unique(bra[idx], axis=0, return_inverse=True)
        uk, ik = np.unique(ket[idx], axis=0, return_inverse=True)
        ib, ik = ib.reshape(-1), ik.reshape(-1)
        levels, gather, n_herm = _r_levels(L), _gather(Lb, Lk), len(_hermite(L))
        per = 8.0 * (Kb * Kk * (hb * hk * 2 + 3 * n_herm + 300) + nb * Kb * hb + Kk * hk * nk + Kb * hb * nk + nb * nk)
        step = max(1, int(limit / per))
        for s in range(0, len(idx), step):
            sel = slice(s, s + step)
            vb, jb = np.unique(ib[sel], return_inverse=True)
            vk, jk = np.unique(ik[sel], return_inverse=True)
            Pb, Pk = _PairSet(bb, cb, ub[vb], False), _PairSet(bk, ck, uk[vk], True)
            jb, jk = torch.as_tensor(jb.reshape(-1), device=dev), torch.as_tensor(jk.reshape(-1), device=dev)
            m = len(jb)
            p, q = Pb.p[jb][:, :, None], Pk.p[jk][:, None, :]
            X = Pb.P[jb][:, :, None] - Pk.P[jk][:, None]                                 # [m, Kb, Kk, 3]
            rho = p * q / (p + q)
            F = _Boys.apply(rho * (X ** 2).sum(-1), L)
            pre = 2.0 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q))
            G = [F[..., n] * pre * (-2.0 * rho) ** n for n in range(L + 1)]
            R = G[L][..., None]
            for N in range(1, L + 1):
                axis, one, two, c = levels[N - 1]
                R = X[..., axis] * R[..., one] + c.to(R.dtype) * R[..., two]
                R = torch.cat([G[L - N][..., None], R[..., 1:]], -1)
            H = R[..., gather].reshape(m, Kb, Kk, hb, hk).transpose(2, 3).reshape(m, Kb * hb, Kk * hk)
            ket_m = Pk.M.transpose(2, 3).reshape(len(vk), Kk * hk, nk)[jk]
            bra_m = Pb.M.transpose(1, 2).reshape(len(vb), nb, Kb * hb)[jb]
            yield idx[sel], torch.bmm(bra_m, torch.bmm(H, ket_m))


def _solid(l):
    """Real solid harmonics m = -l..l over the Cartesian components (the closed form with Racah's normalisation)."""
    at = {c: i for i, c in enumerate(_cart(l))}
    S = np.zeros((2 * l + 1, len(at)))
    for m in range(-l, l + 1):
        a = abs(m)
        norm = math.sqrt((1.0 if m == 0 else 2.0) * math.factorial(l + a) * math.factorial(l - a)) / (2 ** a * math.factorial(l))
        for t in range((l - a) // 2 + 1):
            for u in range(t + 1):
                for w in range(0 if m >= 0 else 1, a + 1, 2):                            # w = 2v
                    c = (-1.0) ** (t + (w - (0 if m >= 0 else 1)) // 2) * 0.25 ** t
                    c *= math.comb(l, t) * math.comb(l - t, a + t) * math.comb(t, u) * math.comb(a, w)
                    S[m + l, at[2 * t + a - 2 * u - w, 2 * u + w, l - 2 * t - a]] += norm * c
    return S


def _centers(bas):
    return torch.as_tensor(bas.center, device="cuda")


def _digest(bas, D, pairs, qp, idx, V, K):
    """K += the four blocks of the unique quartets idx (their transposes are added at the end)."""
    i, j, k, l = pairs[qp[idx, 0], 0], pairs[qp[idx, 0], 1], pairs[qp[idx, 1], 0], pairs[qp[idx, 1], 1]
    w = np.where(i == j, 0.5, 1.0) * np.where(k == l, 0.5, 1.0) * np.where(qp[idx, 0] == qp[idx, 1], 0.5, 1.0)
    nc = [inputs.ncart(int(bas.l[x[0]])) for x in (i, j, k, l)]
    V = V.reshape(-1, *nc) * torch.as_tensor(w, device=V.device)[:, None, None, None, None]
    ao = [torch.as_tensor(bas.ao_off[x], dtype=torch.long, device=V.device)[:, None] + torch.arange(n, device=V.device)
          for x, n in zip((i, j, k, l), nc)]
    blk = lambda x, y: D[ao[x][:, :, None], ao[y][:, None, :]]  # noqa: E731
    for (x, y), (r, s), eq in (((0, 2), (1, 3), "qbd,qabcd->qac"), ((0, 3), (1, 2), "qbc,qabcd->qad"),
                               ((1, 2), (0, 3), "qad,qabcd->qbc"), ((1, 3), (0, 2), "qac,qabcd->qbd")):
        K = K.index_put((ao[x][:, :, None].expand(-1, -1, nc[y]), ao[y][:, None, :].expand(-1, nc[x], -1)),
                        torch.einsum(eq, blk(r, s), V), accumulate=True)
    return K


def _exact_exchange(bas, D, grad):
    """K, and the energy -sum D K with its gradient with respect to the atoms where `grad`."""
    pairs = _pairs(bas.n_shells)
    a, b = np.tril_indices(len(pairs))
    qp = np.stack([a, b], 1)
    D = torch.as_tensor(D, device="cuda")
    atom = torch.as_tensor(bas.atom, dtype=torch.long, device="cuda")
    xyz = torch.as_tensor(bas.atoms, device="cuda")
    K = torch.zeros_like(D)
    g = torch.zeros_like(xyz)
    blocks = lambda c, sel, lim: _blocks(bas, c, bas, c, pairs[qp[sel, 0]], pairs[qp[sel, 1]], lim)  # noqa: E731
    if not grad:
        for idx, V in blocks(xyz[atom], slice(None), 4e9):
            K = _digest(bas, D, pairs, qp, idx, V, K)
        K = K + K.T
        return K, -(D * K).sum(), None
    energy = torch.zeros((), dtype=torch.float64, device="cuda")
    leaf = xyz.clone().requires_grad_()
    with torch.enable_grad():
        gen = blocks(leaf[atom], slice(None), 2e9)
        for idx, V in gen:
            part = -2.0 * (D * _digest(bas, D, pairs, qp, idx, V, torch.zeros_like(D))).sum()
            (d,) = torch.autograd.grad(part, leaf, retain_graph=True)
            g, energy = g + d, energy + part.detach()
    return None, energy, g


def exact(case, seed):
    kind, h = case["kind"], _host_inputs(case, seed)
    with torch.no_grad():
        if kind in ("eri4", "grid4"):
            b, q = h["basis"], h["quartets"]
            cost = np.concatenate([b.l[q], b.nprim[q]], 1)
            if sum(n * _dense_flops(list(map(int, k[:4])), list(map(int, k[4:])))
                   for k, n in zip(*np.unique(cost, axis=0, return_counts=True))) > EXACT_FLOPS:
                return None
            sph = kind == "grid4" and case["sph"]
            nf = 2 * b.l.astype(np.int64) + 1 if sph else (b.l.astype(np.int64) + 1) * (b.l + 2) // 2
            size = nf[q[:, 0]] * nf[q[:, 1]] * nf[q[:, 2]] * nf[q[:, 3]]
            offs = np.concatenate([[0], np.cumsum(size)])
            out = torch.empty(int(offs[-1]), dtype=torch.float64, device="cuda")
            c = _centers(b)
            for idx, V in _blocks(b, c, b, c, q[:, :2], q[:, 2:]):
                l = [int(x) for x in b.l[q[idx[0]]]]
                if sph:
                    V = V.reshape(-1, *[inputs.ncart(x) for x in l])
                    for ax, x in enumerate(l):
                        S = torch.as_tensor(_solid(x), device="cuda")
                        V = torch.movedim(torch.tensordot(V, S, dims=([ax + 1], [1])), -1, ax + 1)
                n = int(size[idx[0]])
                at = torch.as_tensor(offs[idx], device="cuda")[:, None] + torch.arange(n, device="cuda")
                out[at.reshape(-1)] = V.reshape(-1)
            return (out, torch.as_tensor(offs, device="cuda")) if kind == "eri4" else out
        if kind == "df":
            aux, orb, t = h["aux"], h["orb"], h["triplets"]
            nc = lambda b, s: (b.l[s].astype(np.int64) + 1) * (b.l[s] + 2) // 2  # noqa: E731
            size = nc(aux, t[:, 0]) * nc(orb, t[:, 1]) * nc(orb, t[:, 2])
            offs = np.concatenate([[0], np.cumsum(size)])
            out = torch.empty(int(offs[-1]), dtype=torch.float64, device="cuda")
            bra = np.stack([t[:, 0], np.full(len(t), -1)], 1)
            for idx, V in _blocks(aux, _centers(aux), orb, _centers(orb), bra, t[:, 1:]):
                at = torch.as_tensor(offs[idx], device="cuda")[:, None] + torch.arange(V[0].numel(), device="cuda")
                out[at.reshape(-1)] = V.reshape(-1)
            return out
        if kind == "exchange":
            if case["heavy"] + case["light"] > 4:
                return None
            K, e, _ = _exact_exchange(h["basis"], h["D"], False)
            return K, e
        if kind == "gradient":
            if case["heavy"] + case["light"] > 3:
                return None
            _, e, g = _exact_exchange(h["basis"], h["D"], True)
            return g, e
        values, spent = [], 0
        for b, D in zip(h["bases"], h["Ds"]):     # the first molecules that take some seconds together
            spent += b.n_atoms ** 2
            values.append(_exact_exchange(b, D, False)[0] if spent <= 14 else None)
        return values
