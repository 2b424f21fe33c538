"""Timed cases of the library: whole calls through the public entry points, over the sizes users run.

A case is a dict of plain values: a task (which entry point), a basis family with its number of atoms,
and what else the call takes.  The basis families are those of the repository's own workloads:

    plain     atoms with l = 0, 1, 2 shells of three primitives, exponents 0.1 .. 100
    high      atoms with one uncontracted shell per l = 0 .. lmax, exponents 0.05 .. 50
    molecule  40 % hydrogen (3s2p1d), the rest 5s4p3d2f1g, 1 .. 8 primitives, exponents 0.05 .. 5000

``exact`` evaluates the same integrals in 64 bits another way: Cartesian Gaussians, the Laplace form
of 1/r on Gauss-Legendre nodes and Gauss-Hermite sums per Cartesian direction.
"""
import math
import random

import numpy as np
import torch

from paper_2404_16245_gb300 import shgo

H_SHELLS = [0, 0, 0, 1, 1, 2]
HEAVY_SHELLS = [0] * 5 + [1] * 4 + [2] * 3 + [3] * 2 + [4]
PRECISION = {"fp64": shgo.SHGO_PREC_FP64, "fp32": shgo.SHGO_PREC_FP32_BULK}


def listed():
    return [
        # the smallest call: one small molecule's matrix, bound by launches and latency
        {"name": "attraction_small", "task": "attraction", "family": "plain", "atoms": 4, "lmax": 2,
         "precision": "fp64"},
        # the benchmark's call: a 32-atom molecule with shells up to l = 6
        {"name": "attraction_high_l", "task": "attraction", "family": "high", "atoms": 32, "lmax": 6,
         "precision": "fp64"},
        # the same call in the FP32-bulk mode
        {"name": "attraction_high_l_fp32", "task": "attraction", "family": "high", "atoms": 32, "lmax": 6,
         "precision": "fp32"},
        # an ordinary contracted molecule, one call per geometry (an odd number of atoms)
        {"name": "attraction_molecule", "task": "attraction", "family": "molecule", "atoms": 29, "lmax": 4,
         "precision": "fp64"},
        # a set of molecules of mixed sizes in one call, the largest work here
        {"name": "attraction_batch", "task": "batch", "family": "molecule", "atoms": 31, "lmax": 4, "molecules": 6,
         "precision": "fp64"},
        # the potential of a density on a grid of points (a ragged count)
        {"name": "potential_grid", "task": "potential", "family": "high", "atoms": 32, "lmax": 6, "points": 2003},
        # its gradient at the charges of an embedding
        {"name": "potential_gradient", "task": "potential_gradient", "family": "high", "atoms": 32, "lmax": 6,
         "points": 251},
        # derivative matrices by the basis-function centres
        {"name": "derivative_matrices", "task": "derivative", "family": "high", "atoms": 32, "lmax": 6},
        # forces: the same derivatives contracted with a density, contracted molecule
        {"name": "force_molecule", "task": "force", "family": "molecule", "atoms": 17, "lmax": 4},
        # the Coulomb metric of a fitting basis
        {"name": "coulomb_metric", "task": "coulomb", "family": "high", "atoms": 32, "lmax": 6},
        # the overlap matrix
        {"name": "overlap_matrix", "task": "overlap", "family": "high", "atoms": 32, "lmax": 6},
        # all electron-repulsion integrals of a small molecule
        {"name": "repulsion_tensor", "task": "repulsion", "family": "plain", "atoms": 4, "lmax": 2},
    ]


def draw(rng: random.Random):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    task = rng.choice(["attraction", "attraction", "attraction", "batch", "potential", "potential_gradient",
                       "derivative", "force", "coulomb", "overlap", "repulsion", "coulomb_exchange"])
    if task in ("repulsion", "coulomb_exchange"):
        if rng.random() < 0.3:
            return {"task": task, "family": "plain", "atoms": rng.choice([1, 2, 3, 5]), "lmax": rng.randint(1, 2)}
        lmax = rng.randint(1, 3)
        return {"task": task, "family": "high", "atoms": rng.randint(2, {1: 12, 2: 8, 3: 5}[lmax]), "lmax": lmax}
    if task == "batch":
        return {"task": task, "family": "molecule", "atoms": log_int(8, 31), "lmax": 4, "molecules": rng.randint(2, 5),
                "precision": rng.choice(["fp64", "fp32"])}
    if task == "force":
        return {"task": task, "family": "molecule", "atoms": log_int(3, 17), "lmax": 4}
    if task == "attraction":
        family = rng.choice(["plain", "high", "molecule"])
        atoms = {"plain": log_int(3, 60), "high": log_int(2, 40), "molecule": log_int(3, 40)}[family]
        lmax = {"plain": rng.randint(1, 3), "high": rng.randint(2, 6), "molecule": 4}[family]
        return {"task": task, "family": family, "atoms": atoms, "lmax": lmax,
                "precision": rng.choice(["fp64", "fp64", "fp32"])}
    case = {"task": task, "family": "high", "atoms": log_int(3, 32), "lmax": rng.randint(2, 6)}
    if task == "potential":
        case["points"] = log_int(1, 2003)
    if task == "potential_gradient":
        case["points"] = log_int(1, 251)
    return case


# ------------------------------------------------------------------------------------------------ inputs
def _molecule(family, atoms, lmax, rng):
    """(basis dict, centers [n, 3], charges [n]); shells and primitive counts follow from the sizes alone."""
    def log_uniform(lo, hi, n):
        return np.exp(rng.uniform(math.log(lo), math.log(hi), n))

    counts = np.random.default_rng(atoms)
    box = {"plain": 6.0 * (atoms / 4) ** (1 / 3), "high": 20.0 * (atoms / 32) ** (1 / 3),
           "molecule": (atoms / 0.05) ** (1 / 3)}[family]
    xyz = rng.uniform(0.0, box, (atoms, 3))
    l, nprim, exps, coefs, at = [], [], [], [], []
    charges = np.zeros(atoms)
    for a in range(atoms):
        hydrogen = family == "molecule" and a % 5 in (1, 3)
        if family == "molecule":
            charges[a] = 1.0 if hydrogen else float(rng.integers(6, 10))
            shells = H_SHELLS if hydrogen else HEAVY_SHELLS
        else:
            charges[a] = float(rng.integers(1, 9 if family == "plain" else 11))
            shells = range(lmax + 1)
        for ls in shells:
            k = {"plain": 3, "high": 1}.get(family) or int(counts.integers(1, 9))
            lo, hi = {"plain": (0.1, 100.0), "high": (0.05, 50.0), "molecule": (0.05, 5000.0)}[family]
            l.append(ls)
            nprim.append(k)
            exps.extend(log_uniform(lo, hi, k))
            coefs.extend(rng.uniform(0.1, 1.0, k) if k > 1 else [1.0])
            at.append(a)
    basis = {"l": np.asarray(l, dtype=np.int32), "nprim": np.asarray(nprim, dtype=np.int32),
             "exps": np.asarray(exps), "coefs": np.asarray(coefs), "xyz": xyz[at]}
    return basis, xyz, charges


def _inputs(case, seed):
    """Everything of a case on the host: molecules, points and density."""
    rng = np.random.default_rng([int(seed), 77])
    sizes = [case["atoms"]]
    if case["task"] == "batch":  # mixed sizes around the stated one
        sizes = [max(2, int(round(case["atoms"] * f))) for f in (1.0, 0.6, 1.3, 0.4, 0.8, 1.1)[:case["molecules"]]]
    mols = [_molecule(case["family"], n, case["lmax"], rng) for n in sizes]
    basis, xyz, _ = mols[0]
    more = {}
    if "points" in case:  # in and around the molecule, as on a grid or at embedding charges
        more["points"] = rng.uniform(xyz.min(0) - 4.0, xyz.max(0) + 4.0, (case["points"], 3))
    if case["task"] in ("potential", "potential_gradient", "force", "coulomb_exchange"):
        n = int(np.sum(2 * basis["l"] + 1))
        d = rng.standard_normal((n, n)) / n
        more["density"] = (d + d.T) / 2 + np.diag(rng.uniform(0.0, 1.0, n))
    return mols, more


def prepare(case, seed):
    mols, more = _inputs(case, seed)

    def gpu(a):
        return torch.tensor(a, dtype=torch.float64, device="cuda")

    state = {"task": case["task"], **{k: gpu(v) for k, v in more.items()}}
    precision = PRECISION[case.get("precision", "fp64")]
    if case["task"] == "batch":
        state["batch"] = shgo.Batch([(b, len(z)) for b, _, z in mols], precision)
        state["centers"] = gpu(np.concatenate([c for _, c, _ in mols]))
        state["charges"] = gpu(np.concatenate([z for _, _, z in mols]))
    else:
        basis, xyz, charges = mols[0]
        state["basis"] = shgo.Basis(basis, precision)
        state["centers"], state["charges"] = gpu(xyz), gpu(charges)
    return state


def run(state):
    task = state["task"]
    if task == "attraction":
        return shgo.nuclear_attraction(state["basis"], state["centers"], state["charges"])
    if task == "batch":
        return shgo.nuclear_attraction_batched(state["batch"], state["centers"], state["charges"])
    if task == "potential":
        return shgo.esp(state["basis"], state["density"], state["points"])
    if task == "potential_gradient":
        return shgo.esp_gradient(state["basis"], state["density"], state["points"])
    if task == "derivative":
        return shgo.nuclear_attraction_deriv(state["basis"], state["centers"], state["charges"])
    if task == "force":
        return shgo.nuclear_attraction_gradient(state["basis"], state["density"], state["centers"], state["charges"])
    if task == "coulomb":
        return shgo.coulomb_2c(state["basis"])
    if task == "overlap":
        return shgo.overlap(state["basis"])
    if task == "repulsion":
        return shgo.eri(state["basis"])
    if task == "coulomb_exchange":
        return shgo.eri_jk(state["basis"], state["density"])
    raise ValueError(task)


# ------------------------------------------------------------------------------------------------ work
def _live_pairs(basis):
    """{(la, lb): [primitive pairs, shell pairs]} with la >= lb, primitive pairs whose Gaussian product is not
    below 1e-20."""
    prim = _primitives(basis)
    l, e, x, s = prim["l"], prim["exp"], prim["xyz"], prim["shell"]
    found = {}
    for la in range(l.max() + 1):
        for lb in range(la + 1):
            i, j = np.nonzero(l == la)[0], np.nonzero(l == lb)[0]
            r2 = ((x[i][:, None] - x[j][None]) ** 2).sum(-1)
            mu = e[i][:, None] * e[j][None] / (e[i][:, None] + e[j][None])
            live = mu * r2 < 46.0
            if la == lb:
                live &= s[i][:, None] >= s[j][None]
            na, nb = (basis["l"] == la).sum(), (basis["l"] == lb).sum()
            found[la, lb] = [int(live.sum()), int(na * nb if la != lb else na * (na + 1) // 2)]
    return found


def work(case):
    """Least traffic (inputs read once, outputs written once) and the arithmetic of the method (a multiply-add
    counts two): per primitive pair and nucleus (or point) the Boys values, radial factors, harmonics and sums of
    order la + lb, per primitive pair the coupling of its angular parts."""
    def n_r(lam):
        return (lam + 1) * (lam + 2) * (lam + 3) // 6

    mols, more = _inputs(case, 0)
    nbytes = sum(8 * v.size for v in more.values())
    flops = 0
    for basis, xyz, _ in mols:
        n = int(np.sum(2 * basis["l"] + 1))
        pairs = _live_pairs(basis)
        task = case["task"]
        nbytes += 32 * len(xyz) + 16 * len(basis["exps"])
        at = case.get("points", len(xyz))
        nbytes += 8 * {"attraction": n * n, "batch": n * n, "potential": at, "potential_gradient": 3 * at,
                       "derivative": 3 * n * n, "force": 3 * len(basis["l"]), "coulomb": n * n, "overlap": n * n,
                       "repulsion": n ** 4, "coulomb_exchange": 2 * n * n}[task]
        if task in ("repulsion", "coulomb_exchange"):
            quart = list(pairs.items())
            for a, ((la, lb), (pp, _)) in enumerate(quart):
                for (lc, ld), (qq, _) in quart[:a + 1]:
                    half = 0.5 if (la, lb) == (lc, ld) else 1.0
                    r1, r2 = n_r(la + lb), n_r(lc + ld)
                    ncd = (2 * lc + 1) * (2 * ld + 1)
                    flops += half * pp * qq * (2 * r1 * r2 + 2 * r1 * r2 * ncd + 2 * n_r(la + lb + lc + ld))
            continue
        for (la, lb), (pp, sp) in pairs.items():
            up = 1 if task in ("derivative", "force", "potential_gradient") else 0
            lam = la + lb + up
            blk = (2 * la + 1) * (2 * lb + 1)
            if task == "overlap":
                flops += pp * 4 * (lb + 1) + sp * 2 * blk * (2 * lb + 1)
            elif task == "coulomb":
                flops += pp * (100 + 4 * lam) + sp * (2 * blk * (lb + 1) + 4 * (lam + 1) ** 2)
            else:
                per_point = 100 + 4 * (lam + 1) ** 2 + (lam + 2) ** 2 // 2 + 2 * n_r(lam) * (3 if up and "points" in case else 1)
                per_pair = 4 * (la + 1) ** 2 * (lb + 1) ** 2 * (3 if up and "points" not in case else 1)
                flops += pp * (at * per_point + per_pair) + sp * 2 * blk * (2 * la + 2 * lb + 2)
    return {"bytes": int(nbytes), "flops": int(flops)}


# ------------------------------------------------------------------------------------------------ exact values
def _double_factorial(n):
    return math.prod(range(n, 0, -2)) if n > 0 else 1


def _primitives(basis):
    """Primitives with their coefficients in normalised contractions: l, exponent, centre, coefficient, shell."""
    l, first = basis["l"], np.concatenate([[0], np.cumsum(basis["nprim"])])
    coef = np.array(basis["coefs"], dtype=np.float64)
    for s, ls in enumerate(l):
        k = slice(first[s], first[s + 1])
        e = basis["exps"][k]
        self2 = math.pi ** 1.5 * _double_factorial(2 * int(ls) - 1) / 2.0 ** int(ls)
        c = coef[k] * np.sqrt((2 * e) ** (ls + 1.5) / self2)
        s2 = (c[:, None] * c[None] * self2 / (e[:, None] + e[None]) ** (ls + 1.5)).sum()
        coef[k] = c / math.sqrt(s2)
    shell = np.repeat(np.arange(len(l)), basis["nprim"])
    return {"l": l[shell], "exp": np.asarray(basis["exps"]), "xyz": basis["xyz"][shell], "coef": coef, "shell": shell}


def _cartesians(l):
    return [(i, j, l - i - j) for i in range(l, -1, -1) for j in range(l - i, -1, -1)]


def _solid_harmonics(l):
    """[2l + 1, Cartesian monomials of degree l]: the real Racah-normalised solid harmonics, m = -l .. l."""
    def times(p, q):
        out = {}
        for a, x in p.items():
            for b, y in q.items():
                k = (a[0] + b[0], a[1] + b[1], a[2] + b[2])
                out[k] = out.get(k, 0.0) + x * y
        return out

    def plus(p, q, s):
        out = dict(p)
        for k, y in q.items():
            out[k] = out.get(k, 0.0) + s * y
        return out

    x, y, z = {(1, 0, 0): 1.0}, {(0, 1, 0): 1.0}, {(0, 0, 1): 1.0}
    r2 = {(2, 0, 0): 1.0, (0, 2, 0): 1.0, (0, 0, 2): 1.0}
    re, im = [{(0, 0, 0): 1.0}], [{}]  # Re, Im of (x + iy)^m
    for m in range(l):
        re.append(plus(times(x, re[m]), times(y, im[m]), -1.0))
        im.append(plus(times(y, re[m]), times(x, im[m]), 1.0))
    mat = np.zeros((2 * l + 1, len(_cartesians(l))))
    where = {c: k for k, c in enumerate(_cartesians(l))}
    for m in range(l + 1):
        # q_k = r^{k - m} P_k^{(m)}(z / r): q_m = (2m - 1)!!, (k - m + 1) q_{k+1} = (2k + 1) z q_k - (k + m) r^2 q_{k-1}
        prev, cur = {}, {(0, 0, 0): float(_double_factorial(2 * m - 1))}
        for k in range(m, l):
            nxt = times(times(z, cur), {(0, 0, 0): (2 * k + 1) / (k - m + 1)})
            prev, cur = cur, plus(nxt, times(r2, prev), -(k + m) / (k - m + 1))
        norm = math.sqrt((2.0 if m else 1.0) * math.factorial(l - m) / math.factorial(l + m))
        for sign, part in ((1, re[m]), (-1, im[m])):
            if m == 0 and sign < 0:
                continue
            for c, v in times(cur, part).items():
                mat[l + sign * m, where[c]] += norm * v
    return mat


NODES = 36  # Gauss-Legendre nodes of the Laplace form of 1/r


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=_device())


def _hermite(n):
    x, w = np.polynomial.hermite.hermgauss(n)
    return _t(x), _t(w / math.sqrt(math.pi))


def _legendre(n, T):
    """Nodes t and weights on [0, 1] for exp(-T t^2) times a polynomial, per T: [..., n]."""
    x, w = np.polynomial.legendre.leggauss(n)
    top = torch.clamp(7.0 / torch.sqrt(T.clamp(min=1e-300)), max=1.0)[..., None]
    return _t((x + 1) / 2) * top, _t(w / 2) * top


def _powers(d, n):
    """[..., n + 1]: d^0 .. d^n."""
    out = [torch.ones_like(d)]
    for _ in range(n):
        out.append(out[-1] * d)
    return torch.stack(out, -1)


def _cart_index(la, lb, lb_dim):
    """Per Cartesian direction, index of (i, j) in a flattened [.., la_dim, lb_dim] table for every (ca, cb)."""
    a, b = np.array(_cartesians(la)), np.array(_cartesians(lb))
    return [_t((a[:, None, k] * lb_dim + b[None, :, k]).reshape(-1), torch.int64) for k in range(3)]


class _Prims:
    """Primitive pairs (i, j) of two angular momenta, as tensors, with the contracted target functions."""

    def __init__(self, basis):
        p = _primitives(basis)
        self.l = p["l"]
        self.exp, self.xyz, self.coef = _t(p["exp"]), _t(p["xyz"]), _t(p["coef"])
        first = np.concatenate([[0], np.cumsum(2 * basis["l"] + 1)])
        self.nbf = int(first[-1])
        self.first = _t(first[:-1][p["shell"]], torch.int64)
        self.lmax = int(self.l.max())

    def pairs(self, la, lb):
        i, j = _t(np.nonzero(self.l == la)[0], torch.int64), _t(np.nonzero(self.l == lb)[0], torch.int64)
        i, j = i.repeat_interleave(len(j)), j.repeat(len(i))
        a, b = self.exp[i], self.exp[j]
        keep = a * b / (a + b) * ((self.xyz[i] - self.xyz[j]) ** 2).sum(-1) < 60.0
        return i[keep], j[keep]

    def product(self, i, j):
        """p, P, prefactor c_i c_j K_ij of primitive pairs."""
        a, b = self.exp[i], self.exp[j]
        A, B = self.xyz[i], self.xyz[j]
        p = a + b
        P = (a[:, None] * A + b[:, None] * B) / p[:, None]
        return p, P, self.coef[i] * self.coef[j] * torch.exp(-a * b / p * ((A - B) ** 2).sum(-1))


def _attraction_tables(P, i, j, la, lb, centers):
    """Three tables [(la + 1) (lb + 1), pairs, centers * NODES] of one-direction integrals, the weights in the first,
    from the two-index recursion e[i][j+1] = (x - B) e[i][j] + s (i e[i-1][j] + j e[i][j-1])."""
    p, Pc, pref = P.product(i, j)
    d = centers[None] - Pc[:, None]                          # [n, C, 3]
    t, w = _legendre(NODES, p[:, None] * (d ** 2).sum(-1))   # [n, C, q]
    t2 = t * t
    w = w * torch.exp(-(p[:, None] * (d ** 2).sum(-1))[..., None] * t2) * (2 * math.pi / p * pref)[:, None, None]
    s = ((1 - t2).clamp(min=0.0) / (2 * p)[:, None, None]).flatten(1)
    tables = []
    for k in range(3):
        x = (Pc[:, None, None, k] + t2 * d[:, :, None, k]).flatten(1)
        xa, xb = x - P.xyz[i][:, None, k], x - P.xyz[j][:, None, k]
        e = {(0, 0): w.flatten(1) if k == 0 else torch.ones_like(x)}
        for m in range(la):
            e[m + 1, 0] = xa * e[m, 0] + (m * s * e[m - 1, 0] if m else 0)
        for n in range(lb):
            for m in range(la + 1):
                v = xb * e[m, n]
                if m or n:
                    v = v + s * ((m * e[m - 1, n] if m else 0) + (n * e[m, n - 1] if n else 0))
                e[m, n + 1] = v
        tables.append(torch.stack([e[m, n] for m in range(la + 1) for n in range(lb + 1)]))
    return tables


def _chunks(n, cost, most=1.5e8):
    step = max(1, int(most / max(cost, 1)))
    return [slice(k, min(n, k + step)) for k in range(0, n, step)]


def _scatter(out, P, i, j, la, lb, blocks, sa, sb):
    """out[fa, fb] += the Cartesian blocks [n, ca cb] turned into solid harmonics."""
    blk = torch.einsum("ma,nab,kb->nmk", sa, blocks.reshape(len(i), sa.shape[1], sb.shape[1]), sb)
    r = P.first[i][:, None, None] + torch.arange(2 * la + 1, device=blk.device)[None, :, None]
    c = P.first[j][:, None, None] + torch.arange(2 * lb + 1, device=blk.device)[None, None, :]
    out.index_put_((r.expand_as(blk), c.expand_as(blk)), blk, accumulate=True)


def _exact_attraction(basis, xyz, charges):
    P, C, Z = _Prims(basis), _t(xyz), _t(charges)
    out = torch.zeros((P.nbf, P.nbf), dtype=torch.float64, device=_device())
    for la in range(P.lmax + 1):
        for lb in range(la + 1):
            i, j = P.pairs(la, lb)
            sa, sb = _t(_solid_harmonics(la)), _t(_solid_harmonics(lb))
            half = torch.zeros_like(out)
            ix, iy, iz = _cart_index(la, lb, lb + 1)
            for s in _chunks(len(i), len(C) * NODES * len(ix)):
                ex, ey, ez = _attraction_tables(P, i[s], j[s], la, lb, C)
                ex = ex * Z.repeat_interleave(NODES)
                _scatter(half, P, i[s], j[s], la, lb, (ex[ix] * ey[iy] * ez[iz]).sum(2).T, sa, sb)
            out += half if la == lb else half + half.T
    return out


def _by_first(e, exponent, l):
    """Derivative by the first centre of tables [l + 2, ..., pairs, q]: 2 a e[i+1] - i e[i-1]."""
    d = 2 * exponent[:, None] * e[1:]
    for k in range(1, l + 1):
        d[k] -= k * e[k - 1]
    return d


def _exact_derivative(basis, xyz, charges):
    P, C, Z = _Prims(basis), _t(xyz), _t(charges)
    out = torch.zeros((3, P.nbf, P.nbf), dtype=torch.float64, device=_device())
    for la in range(P.lmax + 1):
        for lb in range(P.lmax + 1):
            i, j = P.pairs(la, lb)
            sa, sb = _t(_solid_harmonics(la)), _t(_solid_harmonics(lb))
            idx = _cart_index(la, lb, lb + 1)
            for s in _chunks(len(i), len(C) * NODES * len(idx[0]) * 2):
                tabs = _attraction_tables(P, i[s], j[s], la + 1, lb, C)
                tabs[0] = tabs[0] * Z.repeat_interleave(NODES)
                tabs = [e.unflatten(0, (la + 2, lb + 1)) for e in tabs]
                plain = [e[:la + 1].flatten(0, 1)[k] for e, k in zip(tabs, idx)]
                for x in range(3):
                    v = _by_first(tabs[x], P.exp[i[s]], la).flatten(0, 1)[idx[x]]
                    for y in range(3):
                        if y != x:
                            v = v * plain[y]
                    _scatter(out[x], P, i[s], j[s], la, lb, v.sum(2).T, sa, sb)
    return out


def _exact_potential(basis, density, points, gradient):
    """Values [n], or gradients [n, 3] by d/dC = -(d/dA + d/dB) on the primitives of both centres."""
    P, X, D = _Prims(basis), _t(points), _t(density)
    out = torch.zeros((len(points), 3) if gradient else len(points), dtype=torch.float64, device=_device())
    g = 1 if gradient else 0
    for la in range(P.lmax + 1):
        for lb in range(la + 1):
            i, j = P.pairs(la, lb)
            sa, sb = _t(_solid_harmonics(la)), _t(_solid_harmonics(lb))
            idx = _cart_index(la, lb, lb + 1)
            r = P.first[i][:, None, None] + torch.arange(2 * la + 1, device=_device())[None, :, None]
            c = P.first[j][:, None, None] + torch.arange(2 * lb + 1, device=_device())[None, None, :]
            d = D[r, c] * (1.0 if la == lb else 2.0)  # a symmetric density
            w = torch.einsum("ma,nmk,kb->nab", sa, d, sb).flatten(1)  # in Cartesians
            per = NODES * len(idx[0]) * (8 if gradient else 1)
            npt = max(1, min(len(X), int(1.5e8 / per)))
            for x0 in range(0, len(X), npt):
                pts = X[x0:x0 + npt]
                for s in _chunks(len(i), len(pts) * per):
                    tabs = [e.unflatten(0, (la + g + 1, lb + g + 1)) for e in
                            _attraction_tables(P, i[s], j[s], la + g, lb + g, pts)]
                    plain = [e[:la + 1, :lb + 1].flatten(0, 1)[k] for e, k in zip(tabs, idx)]
                    if not gradient:
                        v = torch.einsum("enq,ne->q", plain[0] * plain[1] * plain[2], w[s])
                        out[x0:x0 + npt] += v.view(len(pts), NODES).sum(1)
                        continue
                    for x in range(3):
                        v = _by_first(tabs[x][:, :lb + 1], P.exp[i[s]], la)
                        v = v + _by_first(tabs[x][:la + 1].transpose(0, 1), P.exp[j[s]], lb).transpose(0, 1)
                        v = -v.flatten(0, 1)[idx[x]]
                        for y in range(3):
                            if y != x:
                                v = v * plain[y]
                        out[x0:x0 + npt, x] += torch.einsum("enq,ne->q", v, w[s]).view(len(pts), NODES).sum(1)
    return out


def _exact_overlap(basis):
    P = _Prims(basis)
    out = torch.zeros((P.nbf, P.nbf), dtype=torch.float64, device=_device())
    for la in range(P.lmax + 1):
        for lb in range(P.lmax + 1):
            i, j = P.pairs(la, lb)
            idx = _cart_index(la, lb, lb + 1)
            h, wh = _hermite((la + lb) // 2 + 1)
            for s in _chunks(len(i), 40 * len(idx[0])):
                p, Pc, pref = P.product(i[s], j[s])
                v = (pref * (math.pi / p) ** 1.5)[:, None]
                for k in range(3):
                    x = Pc[:, k, None] + h / torch.sqrt(p)[:, None]
                    e = torch.einsum("nhi,nhj,h->nij", _powers(x - P.xyz[i[s]][:, k, None], la),
                                     _powers(x - P.xyz[j[s]][:, k, None], lb), wh)
                    v = v * e.flatten(1)[:, idx[k]]
                _scatter(out, P, i[s], j[s], la, lb, v, _t(_solid_harmonics(la)), _t(_solid_harmonics(lb)))
    return out


def _repulsion_tables(p, Pc, q, Qc, A, B, C, D, ls, nodes):
    """Weights [n, t] and [3][n, t, i, j, k, l] one-direction integrals of (x1-A)^i (x1-B)^j (x2-C)^k (x2-D)^l."""
    la, lb, lc, ld = ls
    R = Qc - Pc
    T = p * q / (p + q) * (R ** 2).sum(-1)
    t, w = _legendre(nodes, T)
    t2 = t * t
    w = w * torch.exp(-T[:, None] * t2) * (2 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q)))[:, None]
    sq = t2 / (p + q)[:, None]
    v11 = (1 - t2) / p[:, None] + sq
    s1, s12, s2 = torch.sqrt(v11), sq / torch.sqrt(v11), torch.sqrt((1 - t2).clamp(min=0.0) / ((p * q)[:, None] * v11))
    h1, w1 = _hermite((la + lb + lc + ld) // 2 + 1)
    h2, w2 = _hermite((lc + ld) // 2 + 1)
    tabs = []
    for k in range(3):
        x1 = (Pc[:, None, k] + sq * q[:, None] * R[:, None, k])[..., None] + s1[..., None] * h1
        x2 = ((Qc[:, None, k] - sq * p[:, None] * R[:, None, k])[..., None] + s12[..., None] * h1)[..., None] \
            + s2[..., None, None] * h2
        e1 = torch.einsum("nthi,nthj->nthij", _powers(x1 - A[:, None, None, k], la), _powers(x1 - B[:, None, None, k], lb))
        e2 = torch.einsum("nthgk,nthgl,g->nthkl", _powers(x2 - C[:, None, None, None, k], lc),
                          _powers(x2 - D[:, None, None, None, k], ld), w2)
        tabs.append(torch.einsum("nthij,nthkl,h->ntijkl", e1, e2, w1))
    return w, tabs


def _exact_coulomb(basis):
    P = _Prims(basis)
    out = torch.zeros((P.nbf, P.nbf), dtype=torch.float64, device=_device())
    for la in range(P.lmax + 1):
        for lb in range(P.lmax + 1):
            i, j = (_t(np.nonzero(P.l == k)[0], torch.int64) for k in (la, lb))
            i, j = i.repeat_interleave(len(j)), j.repeat(len(i))
            idx = _cart_index(la, lb, lb + 1)
            for s in _chunks(len(i), 40 * len(idx[0])):
                A, B = P.xyz[i[s]], P.xyz[j[s]]
                w, tabs = _repulsion_tables(P.exp[i[s]], A, P.exp[j[s]], B, A, A, B, B, (la, 0, lb, 0), 40)
                x, y, z = (e.flatten(2)[..., k] for e, k in zip(tabs, idx))
                v = (w[..., None] * x * y * z).sum(1) * (P.coef[i[s]] * P.coef[j[s]])[:, None]
                _scatter(out, P, i[s], j[s], la, lb, v, _t(_solid_harmonics(la)), _t(_solid_harmonics(lb)))
    return out


def _exact_repulsion(basis):
    P = _Prims(basis)
    n = P.nbf
    out = torch.zeros(n ** 4, dtype=torch.float64, device=_device())
    lists = {(la, lb): P.pairs(la, lb) for la in range(P.lmax + 1) for lb in range(la + 1)}
    for (la, lb), (i, j) in lists.items():
        for (lc, ld), (k, l) in lists.items():
            ls = (la, lb, lc, ld)
            dims = [x + 1 for x in ls]
            cart = [np.array(_cartesians(x)) for x in ls]
            idx = []
            for d in range(3):
                g = cart[0][:, None, None, None, d]
                for m in range(1, 4):
                    g = g * dims[m] + cart[m][:, d].reshape([-1 if x == m else 1 for x in range(4)])
                idx.append(_t(g.reshape(-1), torch.int64))
            sph = [_t(_solid_harmonics(x)) for x in ls]
            ab = torch.arange(len(i), device=_device()).repeat_interleave(len(k))
            cd = torch.arange(len(k), device=_device()).repeat(len(i))
            for s in _chunks(len(ab), 30 * len(idx[0])):
                I, J, K, L = i[ab[s]], j[ab[s]], k[cd[s]], l[cd[s]]
                p, Pc, f1 = P.product(I, J)
                q, Qc, f2 = P.product(K, L)
                w, tabs = _repulsion_tables(p, Pc, q, Qc, P.xyz[I], P.xyz[J], P.xyz[K], P.xyz[L], ls, 30)
                x, y, z = (e.flatten(2)[..., g] for e, g in zip(tabs, idx))
                v = torch.einsum("nt,nte->ne", w, x * y * z) * (f1 * f2)[:, None]
                v = v.view(-1, *[len(c) for c in cart])
                v = torch.einsum("nabcd,ma,ob,rc,sd->nmors", v, *sph)
                at = [P.first[f].view(-1, 1, 1, 1, 1) + torch.arange(2 * x + 1, device=_device()).view(
                    [1] + [-1 if m == y else 1 for m in range(4)]) for y, (f, x) in enumerate(zip((I, J, K, L), ls))]
                for a, b in ((0, 1), (1, 0))[:1 if la == lb else 2]:
                    for c, d in ((2, 3), (3, 2))[:1 if lc == ld else 2]:
                        pos = ((at[a] * n + at[b]) * n + at[c]) * n + at[d]
                        out.index_add_(0, pos.expand_as(v).reshape(-1), v.reshape(-1))
    return out.view(n, n, n, n)


def exact(case, seed):
    mols, more = _inputs(case, seed)
    task = case["task"]
    basis, xyz, charges = mols[0]
    if task == "batch":
        out = torch.cat([_exact_attraction(*m).flatten() for m in mols])
    elif task == "attraction":
        out = _exact_attraction(basis, xyz, charges)
    elif task in ("derivative", "force"):
        out = _exact_derivative(basis, xyz, charges)
        if task == "force":
            D = _t(more["density"])
            rows = ((D + D.T)[None] * out).sum(2)  # [3, nbf]
            shell = _t(np.repeat(np.arange(len(basis["l"])), 2 * basis["l"] + 1), torch.int64)
            out = torch.zeros((len(basis["l"]), 3), dtype=torch.float64, device=_device()).index_add_(0, shell, rows.T)
    elif task in ("potential", "potential_gradient"):
        out = _exact_potential(basis, more["density"], more["points"], task == "potential_gradient")
    elif task == "coulomb":
        out = _exact_coulomb(basis)
    elif task == "overlap":
        out = _exact_overlap(basis)
    else:
        out = _exact_repulsion(basis)
        if task == "coulomb_exchange":
            D = _t(more["density"])
            return (torch.einsum("pqrs,rs->pq", out, D), torch.einsum("pqrs,qs->pr", out, D))
    return out
