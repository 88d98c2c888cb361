"""The work a user of the library has it do, as cases that can be timed and checked.

Sizes come from the repository's own workloads (one water / STO-3G, (H2O)_8 and (H2O)_32 / 6-31G*,
linear alkanes C1..C12, the 64-point H2 curve, the learned guess's 2048-row batches):

  jk          one J/K build of a density: a Fock step of a user's own SCF loop (a density on the GPU) or of a
              host program (numpy arrays).  Plain FP64, or the reduced-precision form with its largest
              quartets in double-float, Schwarz threshold 1e-10 (none for the single small molecule).  Such
              a loop builds on the matrices themselves, so the split between FP32 and double-float lies
              where the library puts it for the energy that an SCF reports, 3e-3 (1e-3 for the chains).
  scf         one molecule to self-consistency, Hartree-Fock or Kohn-Sham, in FP64 with tight thresholds.
  scf_batch   many conformers at once, reduced precision, SAD guess: the library's headline batch.
  minimise    the batched dissociation curve by direct minimisation (Adam).
  gradient    SCF energy and analytic nuclear forces of one molecule.
  one_e       overlap, kinetic and nuclear-attraction matrices into device buffers.
  xc          exchange-correlation energy and matrix of a density on the molecular grid.
  mlp         one forward and backward pass of the learned guess's network over host rows.

``exact`` restates each path in 64 bits with plain torch (McMurchie-Davidson Hermite integrals,
autograd for the functional derivatives and the minimiser's gradient); no library code.
"""
import math

import numpy as np
import torch

import mess_inputs as mi
import paper_2406_03121_gb300 as mess

TAU = 1e-10
CUDA = "cuda"


def listed():
    return [
        # the smallest call: one water, minimal basis, host arrays; launches and latency are all of it
        {"name": "jk-water1-sto3g", "kind": "jk", "mol": "water", "n": 1, "basis": "sto-3g", "prec": "fp64",
         "split": 0.0, "tau": 0.0, "host": True},
        # a medium cluster with d shells, both precisions
        {"name": "jk-water8-mixed", "kind": "jk", "mol": "water", "n": 8, "basis": "6-31gs", "prec": "mixed",
         "split": 3e-3, "tau": TAU, "host": False},
        {"name": "jk-water8-fp64", "kind": "jk", "mol": "water", "n": 8, "basis": "6-31gs", "prec": "fp64",
         "split": 0.0, "tau": TAU, "host": False},
        # the library's headline J/K workload: 608 functions
        {"name": "jk-water32-mixed", "kind": "jk", "mol": "water", "n": 32, "basis": "6-31gs", "prec": "mixed",
         "split": 3e-3, "tau": TAU, "host": False},
        # a chain molecule without d shells (95 functions: an odd, ragged size), from host arrays
        {"name": "jk-c7h16-mixed-host", "kind": "jk", "mol": "alkane", "n": 7, "basis": "6-31g", "prec": "mixed",
         "split": 1e-3, "tau": TAU, "host": True},
        # one molecule's Hartree-Fock in plain FP64
        {"name": "scf-c2h6-631gs", "kind": "scf", "mol": "alkane", "n": 2, "basis": "6-31gs", "xc": "hf"},
        # the paper's Kohn-Sham example: CH4, PBE, 6-31G
        {"name": "scf-ch4-pbe", "kind": "scf", "mol": "alkane", "n": 1, "basis": "6-31g", "xc": "pbe"},
        # many conformers in one batch: the largest case
        {"name": "scf-batch-256-mixed", "kind": "scf_batch", "count": 256, "nmin": 1, "nmax": 12},
        # the paper's batched H2 curve: 64 conformers, LDA, 128 Adam steps
        {"name": "minimise-h2x64-lda", "kind": "minimise", "count": 64, "xc": "lda", "steps": 128},
        # energy and forces of one geometry step
        {"name": "gradient-c2h6-631g", "kind": "gradient", "n": 2, "basis": "6-31g"},
        # the one-electron matrices of the headline cluster
        {"name": "one-e-water32", "kind": "one_e", "mol": "water", "n": 32, "basis": "6-31gs"},
        # one training batch of the learned guess
        {"name": "mlp-grad-2048", "kind": "mlp", "rows": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["jk", "jk", "jk", "scf", "scf_batch", "minimise", "gradient", "one_e", "xc", "mlp"])
    basis = rng.choice(["sto-3g", "6-31g", "6-31gs"])
    if kind == "jk":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        mol = rng.choice(["water", "alkane"])
        hi = (8 if prec == "fp64" else 32) if mol == "water" else (4 if prec == "fp64" else 12)
        split = 0.0 if prec == "fp64" else (3e-3 if mol == "water" else 1e-3)
        return {"kind": kind, "mol": mol, "n": _log_int(rng, 1, hi), "basis": basis, "prec": prec, "split": split,
                "tau": rng.choice([TAU, 1e-9, 1e-11]), "host": rng.random() < 0.4}
    if kind == "scf":
        xc = rng.choice(["hf", "hf", "lda", "pbe"])
        return {"kind": kind, "mol": rng.choice(["water", "alkane"]), "n": rng.randint(1, 2) if xc == "hf" else 1,
                "basis": basis, "xc": xc}
    if kind == "scf_batch":
        nmin = rng.randint(1, 6)
        return {"kind": kind, "count": _log_int(rng, 8, 160), "nmin": nmin, "nmax": rng.randint(nmin, 12)}
    if kind == "minimise":
        return {"kind": kind, "count": _log_int(rng, 5, 64), "xc": rng.choice(["hf", "lda", "pbe"]),
                "steps": rng.randint(20, 128)}
    if kind == "gradient":
        return {"kind": kind, "n": rng.randint(1, 3), "basis": rng.choice(["sto-3g", "6-31g"])}
    if kind == "one_e":
        return {"kind": kind, "mol": rng.choice(["water", "alkane"]), "n": _log_int(rng, 1, 12), "basis": basis}
    if kind == "xc":
        return {"kind": kind, "mol": rng.choice(["water", "alkane"]), "n": rng.randint(1, 2), "basis": basis,
                "xc": rng.choice(["lda", "pbe"])}
    return {"kind": kind, "rows": _log_int(rng, 36, 8192)}


# ------------------------------------------------------------------------------------------ inputs
def _molecule(case, seed):
    if case["mol"] == "water":
        return mi.water_cluster(case["n"], 19.0 * (case["n"] / 32.0) ** (1.0 / 3.0), seed)
    return mi.alkane(case["n"], np.random.default_rng(seed))


def _density(mol, basis, seed):
    """A closed-shell-like density: 2 X X^T damped with the distance between the functions' atoms (a
    product of positive semidefinite matrices, so it stays one), as local as a molecule's."""
    cen = np.repeat(np.arange(mol.natom), [sum((l + 1) * (l + 2) // 2 for l, _, _ in _shells_of(z, basis))
                                           for z in mol.Z])
    n = len(cen)
    R = np.linalg.norm(mol.xyz[cen][:, None] - mol.xyz[cen][None], axis=-1)
    D = mi.random_symmetric_density(n, seed, nocc=max(1, mol.nelectron // 2)) * np.exp(-0.4 * R)
    return np.ascontiguousarray(0.5 * (D + D.T))


def _mlp_inputs(rows, seed):
    """Descriptor rows as the network meets them (one-hots, radial basis values in [0, 1]), blocks of a
    minimal-basis density as targets, and the masks of C-C, C-H and H-H pairs."""
    rng = np.random.default_rng(seed)
    X = np.zeros((rows, 112), dtype=np.float32)
    el = rng.integers(0, 2, (rows, 2))
    X[np.arange(rows), el[:, 0]] = 1.0
    X[np.arange(rows), 4 + el[:, 1]] = 1.0
    mu = np.linspace(0.0, 10.0, 32)
    for k in range(3):
        r = rng.uniform(1.5, 20.0, (rows, 1))
        X[:, 9 + 32 * k:41 + 32 * k] = np.exp(-2.0 * (r - mu) ** 2)
    nf = np.where(el == 0, 1, 5)
    M = ((np.arange(5)[None, :, None] < nf[:, 0, None, None]) &
         (np.arange(5)[None, None, :] < nf[:, 1, None, None])).reshape(rows, 25).astype(np.float32)
    T = (0.3 * rng.standard_normal((rows, 25))).astype(np.float32) * M
    fan = np.repeat([112, 112, 256, 256, 256, 256], [112 * 256, 256, 256 * 256, 256, 256 * 32, 32])
    p = (rng.uniform(-1.0, 1.0, fan.size) / np.sqrt(fan)).astype(np.float32)
    return p, X, T, M


def _h2_lengths(case, seed):
    """The dissociation curve's bond lengths, each moved a little by the seed."""
    return np.linspace(0.6, 10.0, case["count"]) + np.random.default_rng(seed).uniform(0.0, 0.05, case["count"])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind in ("jk", "xc", "scf", "one_e"):
        mol = _molecule(case, seed)
        s["basis_set"] = mess.Basis.from_molecule(mol, mi.basis_path(case["basis"]))
    if kind == "jk":
        D = _density(mol, case["basis"], seed)
        s["opts"] = dict(prec=case["prec"], schwarz_tau=case["tau"], fp64_tau=case["split"],
                         split_df32=case["prec"] == "mixed")
        if case["host"]:
            s["D"], s["J"], s["K"] = D, np.zeros_like(D), np.zeros_like(D)
        else:
            s["D"] = torch.from_numpy(D).to(CUDA)
            s["J"], s["K"] = torch.empty_like(s["D"]), torch.empty_like(s["D"])
    elif kind == "xc":
        s["D"] = _density(mol, case["basis"], seed)
    elif kind == "one_e":
        n = s["basis_set"].nbf
        s["out"] = [torch.empty((n, n), dtype=torch.float64, device=CUDA) for _ in range(3)]
    elif kind == "scf_batch":
        s["bases"] = [mess.Basis.from_molecule(m, mi.basis_path("sto-3g"))
                      for m in mi.alkane_batch(case["count"], case["nmin"], case["nmax"], seed)]
    elif kind == "minimise":
        s["bases"] = [mess.Basis.from_molecule(mi.h2(r), mi.basis_path("sto-3g")) for r in _h2_lengths(case, seed)]
    elif kind == "gradient":
        mol = mi.alkane(case["n"], np.random.default_rng(seed))
        s["basis_set"] = mess.Basis.from_molecule(mol, mi.basis_path(case["basis"]))
    elif kind == "mlp":
        p, s["X"], s["T"], s["M"] = _mlp_inputs(case["rows"], seed)
        s["net"] = mess.MLP(seed=1)
        s["net"].set_params(p)
    return s


# ------------------------------------------------------------------------------------------ one pass
ENERGIES = ("E_total", "E_elec", "E_nuc")


def run(s):
    kind = s["kind"]
    if kind == "jk":
        if s["host"]:
            J, K, _ = s["basis_set"].jk(s["D"], J=s["J"], K=s["K"], **s["opts"])
            return [J, K]
        s["basis_set"].jk_device(s["D"], s["J"], s["K"], stream=torch.cuda.current_stream(), **s["opts"])
        return [s["J"], s["K"]]
    if kind == "scf":
        r = s["basis_set"].scf(xc=s["xc"], schwarz_tau=1e-12, conv_E=1e-12, conv_comm=1e-10)
        return [r["D"]] + [r[k] for k in ENERGIES]
    if kind == "scf_batch":
        res, _ = mess.scf_batch(s["bases"], prec="mixed", split_df32=True, guess=mess.MESS_GUESS_SAD,
                                schwarz_tau=TAU)
        return [np.array([r[k] for r in res]) for k in ENERGIES]
    if kind == "minimise":
        res, trace, _ = mess.minimise_batch(s["bases"], xc=s["xc"], steps=s["steps"])
        return [trace] + [np.array([r[k] for r in res]) for k in ENERGIES]
    if kind == "gradient":
        r, g = s["basis_set"].gradient(conv_E=1e-12, conv_comm=1e-10)
        return [g] + [r[k] for k in ENERGIES]
    if kind == "one_e":
        s["basis_set"].one_e_device(*s["out"], stream=torch.cuda.current_stream())
        return s["out"]
    if kind == "xc":
        E, V, _ = s["basis_set"].xc(s["D"], kind=s["xc"])
        return [V, E]
    loss, grad = s["net"].loss_grad(s["X"], s["T"], s["M"])
    return [grad, loss]


# ------------------------------------------------------------------------------------------ work
_SHELL_L = {"S": (0,), "P": (1,), "D": (2,), "SP": (0, 1)}
_FILES = {}


def _shells_of(Z, basis):
    """(l, exponents, file coefficients) of every shell of an element, from the basis data file."""
    if basis not in _FILES:
        data, cur, todo = {}, None, 0
        for line in open(mi.basis_path(basis)):
            tok = line.split("#")[0].split()
            if not tok:
                continue
            if tok[0] == "element":
                cur = data.setdefault(tok[1], [])
            elif todo == 0:
                group = [(l, [], []) for l in _SHELL_L[tok[0].upper()]]
                cur.extend(group)
                todo = int(tok[1])
            else:
                for k, (_, a, c) in enumerate(group):
                    a.append(float(tok[0]))
                    c.append(float(tok[1 + k]))
                todo -= 1
        _FILES[basis] = data
    return _FILES[basis][mi.SYMBOL[int(Z)]]


def _mol_shells(Z, xyz, basis):
    return [(l, np.array(a), np.array(c), np.asarray(R, dtype=float)) for z, R in zip(Z, xyz)
            for l, a, c in _shells_of(z, basis)]


def _function_quartets(mol, basis, tau):
    """Unique Cartesian function quartets, screened by the overlap of the shells' most diffuse primitives."""
    sh = _mol_shells(mol.Z, mol.xyz, basis)
    amin = np.array([a.min() for _, a, _, _ in sh])
    nf = np.array([(l + 1) * (l + 2) // 2 for l, _, _, _ in sh])
    R2 = ((np.array([R for *_, R in sh])[:, None] - np.array([R for *_, R in sh])[None]) ** 2).sum(-1)
    i, j = np.tril_indices(len(sh))
    lq = -(amin[i] * amin[j] / (amin[i] + amin[j])) * R2[i, j]
    w = (nf[i] * nf[j]).astype(float)
    o = np.argsort(lq)
    lq, w = lq[o], w[o]
    tail = np.concatenate([np.cumsum(w[::-1])[::-1], [0.0]])
    cut = np.searchsorted(lq, (math.log(tau) if tau > 0 else -1e300) - lq)
    return 0.5 * float((w * tail[cut]).sum())


def _nbf(mol, basis):
    return sum((l + 1) * (l + 2) // 2 for l, *_ in _mol_shells(mol.Z, mol.xyz, basis))


FLOPS_PER_QUARTET = 30.0   # six FMAs of the digestion, and the recursions of the integral itself


def work(case):
    """Of a typical geometry (a fixed seed): matrices in and out; for the integrals the unique function
    quartets after screening; for an SCF about twelve builds and the eigenproblems."""
    kind = case["kind"]
    if kind == "jk":
        mol = _molecule(case, 1)
        n = _nbf(mol, case["basis"])
        return {"bytes": 24.0 * n * n, "flops": FLOPS_PER_QUARTET * _function_quartets(mol, case["basis"], case["tau"])}
    if kind in ("scf", "gradient"):
        mol = _molecule({"mol": "alkane", **case}, 1)
        n = _nbf(mol, case["basis"])
        pts = sum(512.0 * (50 if z == 1 else 75) for z in mol.Z) if case.get("xc", "hf") != "hf" else 0.0
        q = _function_quartets(mol, case["basis"], 1e-12)
        f = 12.0 * (FLOPS_PER_QUARTET * q + 40.0 * n ** 3 + 4.0 * n * n * pts)
        return {"bytes": 8.0 * n * n, "flops": f + (60.0 * q if kind == "gradient" else 0.0)}
    if kind == "scf_batch":
        f, b = 0.0, 0.0
        for k in range(case["nmin"], case["nmax"] + 1):
            mol = mi.alkane(k, np.random.default_rng(1))
            n = 7 * k + 2
            share = case["count"] / (case["nmax"] - case["nmin"] + 1.0)
            f += share * 12.0 * (FLOPS_PER_QUARTET * _function_quartets(mol, "sto-3g", TAU) + 40.0 * n ** 3)
            b += share * 8.0 * 4.0 * (3 * k + 2)
        return {"bytes": b, "flops": f}
    if kind == "minimise":
        pts = 2 * 50 * 512 if case["xc"] != "hf" else 0
        f = case["count"] * (case["steps"] + 1.0) * (pts * 60.0 + 6 * FLOPS_PER_QUARTET)
        return {"bytes": 8.0 * case["count"] * case["steps"], "flops": f}
    if kind == "one_e":
        mol = _molecule(case, 1)
        n = _nbf(mol, case["basis"])
        return {"bytes": 24.0 * n * n, "flops": 0.5 * n * n * mol.natom * 20.0}
    if kind == "xc":
        mol = _molecule(case, 1)
        n = _nbf(mol, case["basis"])
        pts = sum(512.0 * (50 if z == 1 else 75) for z in mol.Z)
        return {"bytes": 16.0 * n * n, "flops": 4.0 * n * n * pts}
    w = 112 * 256 + 256 * 256 + 256 * 32
    return {"bytes": 4.0 * case["rows"] * (112 + 50) + 8.0 * w, "flops": 6.0 * case["rows"] * w}


# ------------------------------------------------------------------------------------------ in 64 bits
def _t(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64)).to(CUDA)


def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _herm(L):
    return [(t, u, v) for t in range(L + 1) for u in range(L + 1 - t) for v in range(L + 1 - t - u)]


def _odd(k):
    return math.prod(range(k, 0, -2)) if k > 0 else 1


def _boys(nmax, T):
    """F_0..F_nmax: the positive series for F_nmax and the downward recursion below T = 40, erf and the
    upward recursion above."""
    Ts = T.clamp(max=40.0)
    term = torch.full_like(T, 1.0 / (2 * nmax + 1))
    s = term.clone()
    for k in range(1, 170):
        term = term * (2.0 * Ts / (2 * nmax + 2 * k + 1))
        s += term
    e = torch.exp(-Ts)
    lo = [None] * (nmax + 1)
    lo[nmax] = e * s
    for m in range(nmax, 0, -1):
        lo[m - 1] = (2.0 * Ts * lo[m] + e) / (2 * m - 1)
    Tl = T.clamp(min=40.0)
    hi = [0.5 * torch.sqrt(math.pi / Tl) * torch.erf(torch.sqrt(Tl))]
    for m in range(nmax):
        hi.append(((2 * m + 1) * hi[m] - torch.exp(-Tl)) / (2.0 * Tl))
    return [torch.where(T < 40.0, a, b) for a, b in zip(lo, hi)]


def _hermite_r(L, alpha, x, y, z):
    """R_tuv (t + u + v <= L) of the Hermite Coulomb integrals, stacked in the order of _herm(L)."""
    F = _boys(L, alpha * (x * x + y * y + z * z))
    R = {(0, 0, 0, n): F[n] * (-2.0 * alpha) ** n for n in range(L + 1)}
    for N in range(1, L + 1):
        for t, u, v in _herm(N):
            if t + u + v != N:
                continue
            for n in range(L + 1 - N):
                if t:
                    r, a, low = x, (t - 1, u, v), (t - 2, u, v)
                elif u:
                    r, a, low = y, (t, u - 1, v), (t, u - 2, v)
                else:
                    r, a, low = z, (t, u, v - 1), (t, u, v - 2)
                val = r * R[a + (n + 1,)]
                if min(low) >= 0:
                    val = val + ((t or u or v) - 1) * R[low + (n + 1,)]
                R[(t, u, v, n)] = val
    return torch.stack([R[h + (0,)] for h in _herm(L)], dim=-1)


def _e1d(la, lb, a, b, dx):
    """Hermite expansion coefficients E_t^{ij} of one dimension (i <= la, j <= lb), without the
    exponential prefactor: a dict (i, j, t) -> tensor over primitive pairs."""
    p = a + b
    xa, xb, h = -b / p * dx, a / p * dx, 0.5 / p
    E = {(0, 0, 0): torch.ones_like(p)}
    get = lambda i, j, t: E.get((i, j, t), 0.0) if 0 <= t <= i + j and i >= 0 and j >= 0 else 0.0  # noqa: E731
    for i in range(la + 1):
        for j in range(lb + 1):
            for t in range(i + j + 1):
                if i + j == 0:
                    continue
                if i:
                    v = h * get(i - 1, j, t - 1) + xa * get(i - 1, j, t) + (t + 1) * get(i - 1, j, t + 1)
                else:
                    v = h * get(i, j - 1, t - 1) + xb * get(i, j - 1, t) + (t + 1) * get(i, j - 1, t + 1)
                E[(i, j, t)] = v + torch.zeros_like(p)
    return E


class _Exact:
    """The basis of one molecule and its integrals, in 64 bits."""

    def __init__(self, Z, xyz, basis):
        self.Z, self.xyz = np.asarray(Z), np.asarray(xyz, dtype=float)
        self.shells, f0 = [], 0
        for l, a, c, R in _mol_shells(Z, xyz, basis):
            c = c * (2.0 * a / math.pi) ** 0.75 * (4.0 * a) ** (0.5 * l) / math.sqrt(_odd(2 * l - 1))
            p = a[:, None] + a[None]
            c = c / math.sqrt(float((c[:, None] * c[None] * (math.pi / p) ** 1.5 * _odd(2 * l - 1) / (2.0 * p) ** l).sum()))
            self.shells.append((l, a, c, R, f0))
            f0 += (l + 1) * (l + 2) // 2
        self.n = f0
        self.scale = np.concatenate([[math.sqrt(_odd(2 * l - 1) / math.prod(_odd(2 * k - 1) for k in q)) for q in _cart(l)]
                                     for l, *_ in self.shells])
        self.pairs = {}
        for A, sa in enumerate(self.shells):
            for B, sb in enumerate(self.shells[:A + 1]):
                x, y = (sa, sb) if sa[0] >= sb[0] else (sb, sa)
                self.pairs.setdefault((x[0], y[0]), []).append((x, y))
        self.classes = {k: self._class(k, v) for k, v in self.pairs.items()}

    def _class(self, key, pairs):
        la, lb = key
        rows = [(k, al, be, ca * cb, *sa[3], *sb[3]) for k, (sa, sb) in enumerate(pairs)
                for al, ca in zip(sa[1], sa[2]) for be, cb in zip(sb[1], sb[2])]
        own = torch.tensor([r[0] for r in rows], device=CUDA)
        a, b, c, *R = [_t([r[k] for r in rows]) for k in range(1, 10)]
        d = [R[k] - R[3 + k] for k in range(3)]
        p = a + b
        ex = c * torch.exp(-a * b / p * (d[0] ** 2 + d[1] ** 2 + d[2] ** 2))
        e = [_e1d(la, lb + 2, a, b, d[k]) for k in range(3)]
        E = torch.stack([torch.stack([(e[0].get((i[0], j[0], h[0]), 0.0) * torch.ones_like(p))
                                      * e[1].get((i[1], j[1], h[1]), 0.0) * e[2].get((i[2], j[2], h[2]), 0.0) * ex
                                      for h in _herm(la + lb)], -1)
                         for i in _cart(la) for j in _cart(lb)], 1)
        fa, fb = (torch.tensor([s[k][4] for s in pairs], device=CUDA) for k in (0, 1))
        ia = (fa[:, None, None] + torch.arange(len(_cart(la)), device=CUDA)[:, None]).expand(-1, -1, len(_cart(lb))).reshape(len(pairs), -1)
        ib = (fb[:, None, None] + torch.arange(len(_cart(lb)), device=CUDA)[None, :]).expand(-1, len(_cart(la)), -1).reshape(len(pairs), -1)
        sc = _t(self.scale)
        # pairs of different shells stand for both orders
        both = torch.tensor([0.0 if s[0][4] == s[1][4] else 1.0 for s in pairs], dtype=torch.float64, device=CUDA)
        return {"L": la + lb, "la": la, "lb": lb, "own": own, "np": len(pairs), "a": a, "b": b, "p": p, "ex": ex, "e": e,
                "E": E, "P": [(a * R[k] + b * R[3 + k]) / p for k in range(3)], "ia": ia, "ib": ib,
                "sc": sc[ia] * sc[ib], "both": both}

    def _scatter(self, vals):
        """A symmetric matrix from per-class blocks over the pairs' functions."""
        M = torch.zeros(self.n * self.n, dtype=torch.float64, device=CUDA)
        for c, v in zip(self.classes.values(), vals):
            v = v * c["sc"]
            M[(c["ia"] * self.n + c["ib"]).reshape(-1)] = v.reshape(-1)
            M[(c["ib"] * self.n + c["ia"]).reshape(-1)] = v.reshape(-1)
        return M.reshape(self.n, self.n)

    def _sum_pairs(self, c, v):
        return torch.zeros((c["np"],) + v.shape[1:], dtype=torch.float64, device=CUDA).index_add_(0, c["own"], v)

    def one_electron(self):
        S, T, V = [], [], []
        xyz, Z = _t(self.xyz), _t(self.Z)
        for c in self.classes.values():
            w = c["ex"] * (math.pi / c["p"]) ** 1.5
            s = lambda x, i, j: c["e"][x][(i, j, 0)] if i >= 0 and j >= 0 else torch.zeros_like(w)  # noqa: E731
            k1 = lambda x, i, j: (-2.0 * c["b"] ** 2 * s(x, i, j + 2) + c["b"] * (2 * j + 1) * s(x, i, j)  # noqa: E731
                                  - 0.5 * j * (j - 1) * s(x, i, j - 2))
            sv, tv = [], []
            for i in _cart(c["la"]):
                for j in _cart(c["lb"]):
                    o = [s(x, i[x], j[x]) for x in range(3)]
                    k = [k1(x, i[x], j[x]) for x in range(3)]
                    sv.append(w * o[0] * o[1] * o[2])
                    tv.append(w * (k[0] * o[1] * o[2] + o[0] * k[1] * o[2] + o[0] * o[1] * k[2]))
            S.append(self._sum_pairs(c, torch.stack(sv, 1)))
            T.append(self._sum_pairs(c, torch.stack(tv, 1)))
            v = torch.zeros_like(S[-1])
            step = max(1, int(4e7) // (len(self.Z) * 40 * (c["L"] + 1)))
            for q in range(0, len(w), step):
                P = [x[q:q + step, None] - xyz[None, :, k] for k, x in enumerate(c["P"])]
                p = c["p"][q:q + step, None].expand_as(P[0])
                R = (_hermite_r(c["L"], p, *P) * (-Z[None, :, None])).sum(1) * (2.0 * math.pi / p[:, :1])
                v.index_add_(0, c["own"][q:q + step], (c["E"][q:q + step] * R[:, None, :]).sum(-1))
            V.append(v)
        return self._scatter(S), self._scatter(T), self._scatter(V)

    def _integrals(self, x, y):
        """(pairs of x, functions of x, pairs of y, functions of y) repulsion integrals, in slabs of x's pairs."""
        hx, hy = _herm(x["L"]), _herm(y["L"])
        full = {h: k for k, h in enumerate(_herm(x["L"] + y["L"]))}
        idx = torch.tensor([[full[(s[0] + t[0], s[1] + t[1], s[2] + t[2])] for t in hy] for s in hx], device=CUDA)
        sign = _t([(-1.0) ** sum(t) for t in hy])
        Ey = y["E"] * sign
        ends = torch.bincount(x["own"], minlength=x["np"]).cumsum(0).tolist()
        per = len(y["p"]) * max(len(full) * 3, len(hx) * len(hy))
        k0 = 0
        while k0 < x["np"]:
            k1, q0 = k0 + 1, (ends[k0 - 1] if k0 else 0)
            while k1 < x["np"] and (ends[k1] - q0) * per < 6e7:
                k1 += 1
            q1 = ends[k1 - 1]
            p, q = x["p"][q0:q1, None], y["p"][None, :]
            r = [x["P"][k][q0:q1, None] - y["P"][k][None, :] for k in range(3)]
            R = _hermite_r(x["L"] + y["L"], p * q / (p + q), *r) * (2.0 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q)))[..., None]
            R = R[..., idx]                                              # [px, py, hx, hy]
            W = torch.einsum("pqab,qcb->qpac", R, Ey)                    # [py, px, hx, ny]
            W = torch.zeros((y["np"],) + W.shape[1:], dtype=torch.float64, device=CUDA).index_add_(0, y["own"], W)
            W = torch.einsum("ypac,pna->pync", W, x["E"][q0:q1])
            G = torch.zeros((k1 - k0,) + W.shape[1:], dtype=torch.float64, device=CUDA).index_add_(0, x["own"][q0:q1] - k0, W)
            yield k0, k1, G * x["sc"][k0:k1, None, :, None] * y["sc"][None, :, None, :]    # [kx, ky, nx, ny]
            k0 = k1

    def jk(self, D):
        n = self.n
        Jv = [torch.zeros(c["ia"].shape, dtype=torch.float64, device=CUDA) for c in self.classes.values()]
        K = torch.zeros(n * n, dtype=torch.float64, device=CUDA)
        for x, jx in zip(self.classes.values(), Jv):
            for y in self.classes.values():
                Dy = D[y["ia"], y["ib"]] * (1.0 + y["both"])[:, None]
                for k0, k1, G in self._integrals(x, y):
                    jx[k0:k1] += torch.einsum("xyab,yb->xa", G, Dy)
                    ia, ib, bx = x["ia"][k0:k1], x["ib"][k0:k1], x["both"][k0:k1]
                    for a, b, wx in ((ia, ib, torch.ones_like(bx)), (ib, ia, bx)):
                        for c, d, wy in ((y["ia"], y["ib"], torch.ones_like(y["both"])), (y["ib"], y["ia"], y["both"])):
                            at = a[:, None, :, None] * n + c[None, :, None, :]
                            val = G * D[b[:, None, :, None], d[None, :, None, :]] * (wx[:, None] * wy[None])[..., None, None]
                            K.index_add_(0, at.reshape(-1), val.reshape(-1))
        M = torch.zeros(n, n, dtype=torch.float64, device=CUDA)
        for c, v in zip(self.classes.values(), Jv):
            M[c["ia"], c["ib"]] = v
            M[c["ib"], c["ia"]] = v
        return M, K.reshape(n, n)

    def eri(self):
        n = self.n
        T = torch.zeros(n, n, n, n, dtype=torch.float64, device=CUDA)
        for x in self.classes.values():
            for y in self.classes.values():
                for k0, k1, G in self._integrals(x, y):
                    a, b = x["ia"][k0:k1, None, :, None], x["ib"][k0:k1, None, :, None]
                    c, d = y["ia"][None, :, None, :], y["ib"][None, :, None, :]
                    for i, j in ((a, b), (b, a)):
                        T[i, j, c, d] = G
                        T[i, j, d, c] = G
        return T

    def e_nuc(self):
        Z, R = self.Z.astype(float), np.linalg.norm(self.xyz[:, None] - self.xyz[None], axis=-1)
        i, j = np.tril_indices(len(Z), -1)
        return float((Z[i] * Z[j] / R[i, j]).sum())

    def grid(self):
        """Atom-centred points and Becke weights, and every function's value and gradient there."""
        ct, wt = np.polynomial.legendre.leggauss(16)
        ph = 2.0 * math.pi * np.arange(32) / 32
        st = np.sqrt(1.0 - ct ** 2)
        u = np.stack([(st[:, None] * np.cos(ph)).ravel(), (st[:, None] * np.sin(ph)).ravel(), np.repeat(ct, 32)], -1)
        pts, w, own = [], [], []
        for k, (z, R) in enumerate(zip(self.Z, self.xyz)):
            N = 50 if z == 1 else 75
            rad = {1: 0.35, 6: 0.35, 7: 0.325, 8: 0.30}.get(int(z), 0.35) / 0.52917721092
            th = np.arange(1, N + 1) * math.pi / (N + 1)
            x = np.cos(th)
            r = rad * (1 + x) / (1 - x)
            wr = math.pi / (N + 1) * np.sin(th) ** 2 / np.sqrt(1 - x ** 2) * r ** 2 * 2 * rad / (1 - x) ** 2
            pts.append((r[:, None, None] * u + R).reshape(-1, 3))
            w.append((wr[:, None] * np.repeat(wt, 32) * 2.0 * math.pi / 32).ravel())
            own.append(np.full(N * 512, k))
        pts, w, own = _t(np.concatenate(pts)), _t(np.concatenate(w)), torch.as_tensor(np.concatenate(own)).to(CUDA)
        if len(self.Z) > 1:
            d = torch.cdist(pts, _t(self.xyz), compute_mode="donot_use_mm_for_euclid_dist")
            RAB = torch.cdist(_t(self.xyz), _t(self.xyz), compute_mode="donot_use_mm_for_euclid_dist")
            P = torch.ones_like(d)
            for A in range(len(self.Z)):
                for B in range(len(self.Z)):
                    if A != B:
                        f = (d[:, A] - d[:, B]) / RAB[A, B]
                        for _ in range(3):
                            f = 1.5 * f - 0.5 * f ** 3
                        P[:, A] *= 0.5 * (1.0 - f)
            w = w * P.gather(1, own[:, None])[:, 0] / P.sum(1)
        vals, grads = [], []
        for l, a, c, R, _ in self.shells:
            X = pts - _t(R)
            e = torch.exp(-_t(a) * (X ** 2).sum(-1, keepdim=True)) * _t(c)
            g, gd = e.sum(-1), (-2.0 * _t(a) * e).sum(-1)
            for q in _cart(l):
                pw = [X[:, k] ** q[k] for k in range(3)]
                dp = [q[k] * X[:, k] ** max(q[k] - 1, 0) for k in range(3)]
                poly = pw[0] * pw[1] * pw[2]
                vals.append(poly * g)
                grads.append(torch.stack([dp[0] * pw[1] * pw[2] * g + poly * gd * X[:, 0],
                                          pw[0] * dp[1] * pw[2] * g + poly * gd * X[:, 1],
                                          pw[0] * pw[1] * dp[2] * g + poly * gd * X[:, 2]]))
        sc = _t(self.scale)
        return w, torch.stack(vals, 1) * sc, torch.stack(grads, 2) * sc


def _exc(kind, D, w, phi, dphi):
    """E_xc of a density matrix, or of each of a stack of them (differentiable): Slater + Perdew-Wang 1992, or PBE."""
    t = phi @ D
    rho = (t * phi).sum(-1)
    w = torch.where(rho > 1e-14, w, 0.0)      # points with less density carry nothing
    rho = rho.clamp(min=1e-14)
    c = rho ** (1.0 / 3.0)
    ex = -0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * rho * c
    rs = (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0) / c
    A, a1, b1, b2, b3, b4 = 0.031091, 0.21370, 7.5957, 3.5876, 1.6382, 0.49294
    s = torch.sqrt(rs)
    ec = -2.0 * A * (1.0 + a1 * rs) * torch.log1p(1.0 / (2.0 * A * (b1 * s + b2 * rs + b3 * rs * s + b4 * rs * rs)))
    if kind == "lda":
        return (w * (ex + rho * ec)).sum(-1)
    sigma = sum((2.0 * (t * d).sum(-1)) ** 2 for d in dphi)
    kF = (3.0 * math.pi ** 2) ** (1.0 / 3.0) * c
    kappa, beta = 0.804, 0.06672455060314922
    mu, gamma = beta * math.pi ** 2 / 3.0, (1.0 - math.log(2.0)) / math.pi ** 2
    Fx = 1.0 + kappa - kappa / (1.0 + mu * sigma / (4.0 * kF ** 2 * rho ** 2) / kappa)
    u = sigma * math.pi / (16.0 * kF * rho ** 2)
    Ag = beta / gamma / torch.expm1(-ec / gamma)
    H = gamma * torch.log1p(beta / gamma * u * (1.0 + Ag * u) / (1.0 + Ag * u + Ag * Ag * u * u))
    return (w * (ex * Fx + rho * (ec + H))).sum(-1)


def _vxc(kind, D, grid):
    D = D.detach().clone().requires_grad_(True)
    E = _exc(kind, D, *grid)
    (V,) = torch.autograd.grad(E, D)
    return float(E.detach()), 0.5 * (V + V.T)


def _scf_exact(x, xc):
    """The self-consistent density and energies: Roothaan iterations with DIIS over the dense integrals."""
    S, T, V = x.one_electron()
    H, G = T + V, x.eri()
    n, nocc = x.n, int(x.Z.sum()) // 2
    grid = x.grid() if xc != "hf" else None
    s, U = torch.linalg.eigh(S)
    X = U @ torch.diag(s ** -0.5) @ U.T

    def dens(F):
        C = X @ torch.linalg.eigh(X @ F @ X)[1][:, :nocc]
        return 2.0 * C @ C.T

    def fock(D):
        J = (G.reshape(n * n, n * n) @ D.reshape(-1)).reshape(n, n)
        if xc == "hf":
            F = H + J - 0.5 * torch.einsum("mlns,ls->mn", G, D)
            return F, 0.5 * float((D * (H + F)).sum())
        E, Vx = _vxc(xc, D, grid)
        return H + J + Vx, float((D * (H + 0.5 * J)).sum()) + E

    D, Fs, es = dens(H), [], []
    for _ in range(120):
        F, E = fock(D)
        e = F @ D @ S - S @ D @ F
        if float(e.abs().max()) < 2e-12 * max(1.0, float(F.abs().max())) and len(es) > 3:
            break
        Fs, es = (Fs + [F])[-8:], (es + [X @ e @ X])[-8:]
        k = len(Fs)
        B = -np.ones((k + 1, k + 1))
        B[:k, :k] = [[float((p * q).sum()) for q in es] for p in es]
        B[k, k] = 0.0
        sc = B[:k, :k].diagonal().max()
        B[:k, :k] /= sc
        c = np.linalg.lstsq(B, np.r_[np.zeros(k), -1.0], rcond=None)[0][:k]
        D = dens(sum(ci * Fi for ci, Fi in zip(c, Fs)))
    return D, E


def _minimise_exact(case, seed):
    mols = [mi.h2(r) for r in _h2_lengths(case, seed)]
    xs = [_Exact(m.Z, m.xyz, "sto-3g") for m in mols]
    S, H, G, X = [], [], [], []
    for x in xs:
        s, t, v = x.one_electron()
        S.append(s)
        H.append(t + v)
        G.append(x.eri())
        w, U = torch.linalg.eigh(s)
        X.append(U @ torch.diag(w ** -0.5) @ U.T)
    H, G, X = torch.stack(H), torch.stack(G), torch.stack(X)
    grids = [x.grid() for x in xs] if case["xc"] != "hf" else None
    if grids:
        w, phi, dphi = (torch.stack([g[k] for g in grids]) for k in range(3))
        dphi = dphi.transpose(0, 1)
    enuc = _t([x.e_nuc() for x in xs])

    def energies(Z):
        q = Z[:, :, 0] / Z[:, :, 0].norm(dim=1, keepdim=True)     # the first column of Q: the occupied one
        C = (X @ q[:, :, None])[:, :, 0]
        D = 2.0 * C[:, :, None] * C[:, None, :]
        J = torch.einsum("bmnls,bls->bmn", G, D)
        if grids is None:
            K = torch.einsum("bmlns,bls->bmn", G, D)
            return (D * (H + 0.5 * J - 0.25 * K)).sum((1, 2)) + enuc
        return (D * (H + 0.5 * J)).sum((1, 2)) + enuc + _exc(case["xc"], D, w, phi, dphi)

    Z = torch.eye(2, dtype=torch.float64, device=CUDA).repeat(len(xs), 1, 1)
    m, v, trace = torch.zeros_like(Z), torch.zeros_like(Z), []
    for t in range(1, case["steps"] + 1):
        Z = Z.detach().requires_grad_(True)
        E = energies(Z)
        (g,) = torch.autograd.grad(E.sum(), Z)
        trace.append(E.detach())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        Z = Z.detach() - 0.1 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    E = energies(Z).detach()
    return [torch.stack(trace), E, E - enuc, enuc]


EXACT_JK_FUNCTIONS, EXACT_ERI_FUNCTIONS = 160, 48    # what the dense sums reach within about 20 seconds


def exact(case, seed):
    kind = case["kind"]
    if kind == "scf_batch":
        return None                    # hundreds of molecules' dense integrals
    if kind == "minimise":
        return _minimise_exact(case, seed)
    if kind == "mlp":
        p, *rows = _mlp_inputs(case["rows"], seed)
        X, T, M = (_t(r) for r in rows)
        p = _t(p).requires_grad_(True)
        W1, b1, W2, b2, W3, b3 = torch.split(p, [112 * 256, 256, 256 * 256, 256, 256 * 32, 32])
        h = torch.nn.functional.silu(X @ W1.reshape(112, 256) + b1)
        h = torch.nn.functional.silu(h @ W2.reshape(256, 256) + b2)
        y = (h @ W3.reshape(256, 32) + b3)[:, :25]
        loss = (M * (y - T) ** 2).sum() / M.sum()
        return [torch.autograd.grad(loss, p)[0], float(loss.detach())]
    mol = mi.alkane(case["n"], np.random.default_rng(seed)) if kind == "gradient" else _molecule(case, seed)
    n = _nbf(mol, case["basis"])
    if (kind == "jk" and n > EXACT_JK_FUNCTIONS) or (kind in ("scf", "gradient") and n > EXACT_ERI_FUNCTIONS):
        return None
    x = _Exact(mol.Z, mol.xyz, case["basis"])
    if kind == "jk":
        return list(x.jk(_t(_density(mol, case["basis"], seed))))
    if kind == "one_e":
        return list(x.one_electron())
    if kind == "xc":
        E, V = _vxc(case["xc"], _t(_density(mol, case["basis"], seed)), x.grid())
        return [V, E]
    D, E = _scf_exact(x, case.get("xc", "hf"))
    energies = [E + x.e_nuc(), E, x.e_nuc()]
    return [D if kind == "scf" else None] + energies
