"""Measured cases of the C-PCM library: what its users call, over the sizes they call it with.

A quantum-chemistry program calls the library in a few ways:

* once per geometry ("step"): surface, basis set-up, then one SCF iteration's worth of calls;
* once per SCF iteration at a fixed geometry ("scf"): the potential of the new density, the charges to the
  iteration's threshold, the Fock correction and the energy;
* once per geometry-optimisation step ("opt"): a step and the nuclear gradient;
* single calls inside those ("esp", "solve", "fock", "gradient");
* many small molecules at a time ("batch").

PCM_FP64 is the default precision and the one that results are checked in; PCM_MIXED is the fast one.  The
molecules are branching random walks with the elements H:C:N:O:S = 50:31:9:9:1 and 6-31G-like shells (optionally
a d shell per heavy atom), of 3 to 1000 atoms.
"""
import math

import numpy as np
import torch

import paper_1505_07851_gb300 as pcm

EPS, ZETA, NPTS, DROP = 78.39, 4.9, 110, 1e-8     # the library's defaults
F_EPS = (EPS - 1.0) / EPS
BOHR = 1.0 / 0.529177210903
BONDI = {"H": 1.20, "C": 1.70, "N": 1.55, "O": 1.52, "S": 1.80}
CHARGE = {"H": 1, "C": 6, "N": 7, "O": 8, "S": 16}
# (shell l, -1 = sp; primitives; exponent range)
SHELLS = {
    "H": [(0, 3, (0.3, 30.0)), (0, 1, (0.1, 0.4))],
    "C": [(0, 6, (3.0, 5000.0)), (-1, 3, (0.3, 30.0)), (-1, 1, (0.1, 0.4))],
    "N": [(0, 6, (3.0, 5000.0)), (-1, 3, (0.3, 30.0)), (-1, 1, (0.1, 0.4))],
    "O": [(0, 6, (3.0, 5000.0)), (-1, 3, (0.3, 30.0)), (-1, 1, (0.1, 0.4))],
    "S": [(0, 6, (10.0, 5000.0)), (-1, 6, (1.0, 500.0)), (-1, 3, (0.2, 5.0)), (-1, 1, (0.1, 0.4))],
}
WATER_SHELLS = {"H": [(0, 3, (0.1, 130.0))], "O": [(0, 3, (0.1, 130.0)), (-1, 3, (0.1, 130.0))]}
D_SHELL = (2, 1, (0.3, 1.5))


def _case(name, call, natom, d, precision, diis=1e-3, host=False, nmol=0):
    return {"name": name, "call": call, "natom": natom, "d_shells": d, "precision": precision, "diis": diis,
            "host": host, "nmol": nmol}


def listed():
    return [
        # a first call: water with host arrays, all of it (surface to energy); launches and latency
        _case("step3_fp64", "step", 3, False, "fp64", host=True),
        # one optimisation step of a small organic molecule with polarisation functions, host arrays
        _case("opt20_spd_fp64", "opt", 20, True, "fp64", host=True),
        # an SCF iteration of a drug-sized molecule on the device, late in the SCF (tight threshold)
        _case("scf40_sp_mixed", "scf", 40, False, "mixed", diis=1e-5),
        # the potential alone, with d shells (all six shell-pair classes)
        _case("esp100_spd_fp64", "esp", 100, True, "fp64"),
        # the nuclear gradient alone, all terms
        _case("gradient100_spd_fp64", "gradient", 100, True, "fp64"),
        # the Fock correction alone, s and p shells
        _case("fock150_sp_fp64", "fock", 150, False, "fp64"),
        # an SCF iteration of a small protein in FP64
        _case("scf300_sp_fp64", "scf", 300, False, "fp64"),
        # its linear system alone, to the threshold of a converged SCF
        _case("solve300_sp_fp64", "solve", 300, False, "fp64", diis=1e-7),
        # a new geometry of the same protein in mixed precision
        _case("step300_sp_mixed", "step", 300, False, "mixed"),
        # its gradient with d shells
        _case("gradient300_spd_mixed", "gradient", 300, True, "mixed"),
        # the largest protein: 1000 atoms with d shells, a new geometry in mixed precision
        _case("step1000_spd_mixed", "step", 1000, True, "mixed"),
        # conformations of a peptide, eight at a time
        _case("batch8_sp_mixed", "batch", 180, False, "mixed", nmol=8),
    ]


def draw(rng):
    precision = rng.choice(["fp64", "fp64", "mixed"])
    call = rng.choice(["step", "scf", "opt", "esp", "fock", "solve", "gradient"] + (["batch"] if precision == "mixed" else []))
    d = rng.random() < 0.5
    host = rng.random() < 0.25
    if precision == "mixed":
        top = {"batch": 220, "gradient": 600, "opt": 600}.get(call, 1000)
    else:
        top = {"step": 270, "scf": 270, "opt": 120, "gradient": 180}.get(call, 300)
    natom = int(round(math.exp(rng.uniform(math.log(4), math.log(top)))))
    nmol = rng.randint(2, 8) if call == "batch" else 0
    diis = 10.0 ** rng.uniform(-7.0, -2.0)
    c = _case("", call, natom, d, precision, diis=diis, host=host and call != "batch", nmol=nmol)
    del c["name"]
    return c


# -- molecules -----------------------------------------------------------------------------------------------------
class Mol:
    def __init__(self, symbols, xyz):
        self.symbols = symbols
        self.xyz = np.ascontiguousarray(xyz, np.float64)
        self.Z = np.array([CHARGE[s] for s in symbols], np.float64)
        self.radius = np.array([1.2 * BONDI[s] * BOHR for s in symbols])
        self.natom = len(symbols)


class Basis:
    def __init__(self, symbols, shells, d_shells, rng):
        sa, sl, sn, ex, co = [], [], [], [], []
        for a, s in enumerate(symbols):
            for l, n, (lo, hi) in shells[s] + ([D_SHELL] if d_shells and s != "H" else []):
                e = np.sort(np.exp(rng.uniform(math.log(lo), math.log(hi), n)))[::-1]
                sa.append(a), sl.append(l), sn.append(n), ex.extend(e)
                co.extend(rng.uniform(0.1, 1.0, 2 * n if l < 0 else n))
        self.shell_atom, self.shell_l, self.shell_nprim = (np.array(v, np.int32) for v in (sa, sl, sn))
        self.exps, self.coefs = np.array(ex), np.array(co)
        self.nbf = int(sum({0: 1, 1: 3, 2: 6, -1: 4}[l] for l in sl))


def _walk(natom, radius, rng):
    """Bonds of 1.0-1.5 angstrom to a parent (mostly the last atom), at least 2.0 to all others, in a globule."""
    pos = np.zeros((natom, 3))
    n = 1
    while n < natom:
        parent = np.where(rng.random(64) < 0.7, n - 1, rng.integers(0, n, 64))
        v = rng.standard_normal((64, 3))
        cand = pos[parent] + v / np.linalg.norm(v, axis=1)[:, None] * rng.uniform(1.0, 1.5, 64)[:, None]
        dist = np.linalg.norm(cand[:, None, :] - pos[None, :n, :], axis=2)
        dist[np.arange(64), parent] = np.inf
        good = np.flatnonzero((np.linalg.norm(cand, axis=1) <= radius) & np.all(dist >= 2.0, axis=1))
        if len(good):
            pos[n] = cand[good[0]]
            n += 1
    return pos


def _molecule(natom, d_shells, seed):
    """The molecule's shape goes by its size, so that its surface has as many points whatever the seed; the seed gives its
    place, its exponents and its coefficients."""
    shape, rng = np.random.default_rng([natom, 1505]), np.random.default_rng([natom, int(d_shells), seed])
    at = rng.uniform(-4.0, 4.0, 3)
    if natom == 3:
        mol = Mol(["O", "H", "H"], np.array([[0, 0, 0], [1.43, 1.11, 0], [-1.43, 1.11, 0]]) + at)
        return mol, Basis(mol.symbols, WATER_SHELLS, d_shells, rng)
    counts = [int(round(natom * r)) for r in (0.50, 0.31, 0.09, 0.09, 0.01)]
    counts[0] += natom - sum(counts)
    symbols = [s for s, c in zip("HCNOS", counts) for _ in range(c)]
    shape.shuffle(symbols)
    radius = max(3.0, 8.0 * (natom / 300.0) ** (1.0 / 3.0 if natom <= 300 else 0.4346))
    mol = Mol(symbols, _walk(natom, radius, shape) * BOHR + at)
    return mol, Basis(symbols, SHELLS, d_shells, rng)


# -- plain FP64 torch: Gaussian pairs, Hermite expansions, Boys function -----------------------------------------------
def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _herm(L):
    return [(t, u, n - t - u) for n in range(L + 1) for t in range(n, -1, -1) for u in range(n - t, -1, -1)]


def _factor(c):
    return math.sqrt(3.0) if max(c) == 1 and sum(c) == 2 else 1.0


def _prims(basis):
    """{l: (exponents, normalised coefficients, atoms, first basis functions)} on the GPU."""
    got = {l: ([], [], [], []) for l in range(3)}
    off = cp = bf = 0
    for a, l, n in zip(basis.shell_atom, basis.shell_l, basis.shell_nprim):
        e = basis.exps[off:off + n]
        for ll, c in ([(0, basis.coefs[cp:cp + n]), (1, basis.coefs[cp + n:cp + 2 * n])] if l < 0 else [(int(l), basis.coefs[cp:cp + n])]):
            norm = c * (2 * e / np.pi) ** 0.75 * (4 * e) ** (ll / 2) / math.sqrt([1, 1, 3][ll])
            for v, x in zip(got[ll], (e, norm, [a] * n, [bf] * n)):
                v.extend(x)
            bf += len(_cart(ll))
        off += n
        cp += 2 * n if l < 0 else n
    return {l: tuple(torch.tensor(np.array(x), device="cuda", dtype=torch.float64 if i < 2 else torch.int64) for i, x in enumerate(v)) for l, v in got.items()}


def _pairs(prims, xyz, cut, most):
    """Chunks (la, lb, i, j, w) of primitive pairs above `cut`, i of shell l = la and j of lb <= la; w: 2 for pairs that
    stand for their mirror image too."""
    for la in range(3):
        for lb in range(la + 1):
            ea, ca, aa, _ = prims[la]
            eb, cb, ab, _ = prims[lb]
            if not len(ea) or not len(eb):
                continue
            step = max(1, 20_000_000 // len(eb))
            for s in range(0, len(ea), step):
                a, b = ea[s:s + step, None], eb[None, :]
                d2 = (xyz[aa[s:s + step], None, :] - xyz[ab][None, :, :]).square().sum(-1)
                q = (ca[s:s + step, None] * cb[None, :]).abs() * torch.exp(-a * b / (a + b) * d2) / (a + b) ** 1.25
                i, j = torch.nonzero(q > cut, as_tuple=True)
                i = i + s
                if la == lb:
                    i, j = i[i >= j], j[i >= j]
                w = torch.where((i == j) & (la == lb), 1.0, 2.0).double()
                for k in range(0, len(i), most):
                    yield la, lb, i[k:k + most], j[k:k + most], w[k:k + most]


def _expansion(prims, xyz, la, lb, i, j):
    """p, the centre P, c_a c_b K, and E[d][(i, j, t)] (Hermite coefficients, d = x, y, z) of a chunk of pairs."""
    a, b = prims[la][0][i], prims[lb][0][j]
    A, B = xyz[prims[la][2][i]], xyz[prims[lb][2][j]]
    p = a + b
    P = (a[:, None] * A + b[:, None] * B) / p[:, None]
    K = prims[la][1][i] * prims[lb][1][j] * torch.exp(-a * b / p * (A - B).square().sum(-1))
    E = []
    for d in range(3):
        x, y, h = P[:, d] - A[:, d], P[:, d] - B[:, d], 0.5 / p
        e = {(0, 0, 0): torch.ones_like(p)}
        for m in range(la + 1):
            for n in range(lb + 1):
                if m + n == 0:
                    continue
                f, v, (r, s) = (x, None, (m - 1, n)) if m > 0 else (y, None, (m, n - 1))
                for t in range(m + n + 1):
                    v = 0.0
                    if (r, s, t) in e:
                        v = v + f * e[r, s, t]
                    if t > 0 and (r, s, t - 1) in e:
                        v = v + h * e[r, s, t - 1]
                    if (r, s, t + 1) in e:
                        v = v + (t + 1) * e[r, s, t + 1]
                    e[m, n, t] = v
        E.append(e)
    return p, P, K, E


def _blocks(prims, la, lb, i, j):
    """(a, b, factor, rows, columns): the Cartesian components of a chunk of pairs and their basis functions."""
    for u, a in enumerate(_cart(la)):
        for v, b in enumerate(_cart(lb)):
            yield a, b, _factor(a) * _factor(b), prims[la][3][i] + u, prims[lb][3][j] + v


def _product(E, a, b, t):
    """E_t^{ab}, or None where it vanishes."""
    if any(t[d] > a[d] + b[d] for d in range(3)):
        return None
    return E[0][a[0], b[0], t[0]] * E[1][a[1], b[1], t[1]] * E[2][a[2], b[2], t[2]]


def _density(basis, xyz, nocc, gen):
    """P = 2 C C^T with seeded orbitals C orthonormal in the overlap metric."""
    prims = _prims(basis)
    n = basis.nbf
    S = torch.zeros(n * n, dtype=torch.int64, device="cuda")   # fixed point: the same sums in any order
    for la, lb, i, j, w in _pairs(prims, xyz, 1e-14, 4_000_000):
        p, _, K, E = _expansion(prims, xyz, la, lb, i, j)
        for a, b, f, row, col in _blocks(prims, la, lb, i, j):
            v = f * K * (math.pi / p) ** 1.5 * _product(E, a, b, (0, 0, 0))
            # a pair within one shell block is listed once (i >= j): its mirror image is added below
            v = torch.where((w > 1) if la == lb else (w > 0), v, 0.5 * v)
            S.index_add_(0, row * n + col, torch.round(v * 2.0 ** 48).long())
    S = S.view(n, n).double() * 2.0 ** -48
    S = S + S.T
    G = torch.randn(n, nocc, dtype=torch.float64, device="cuda", generator=gen)
    L = torch.linalg.cholesky(G.T @ (S @ G))
    C = torch.linalg.solve_triangular(L, G.T, upper=False).T
    P = 2.0 * C @ C.T
    return (0.5 * (P + P.T)).contiguous()


_TABLE = []


def _boys(m, T):
    """F_0 .. F_m: F_m from a table of series values and a Taylor step (its asymptotic form beyond T = 48), the lower ones
    by downward recursion."""
    if not _TABLE:
        t = np.arange(48 * 32 + 2) / 32.0
        F = np.empty((len(t), 16))
        term = np.full(len(t), 1.0 / 31.0)
        tot = term.copy()
        for k in range(1, 400):
            term = term * 2 * t / (31.0 + 2 * k)
            tot = tot + term
        F[:, 15] = np.exp(-t) * tot
        for k in range(15, 0, -1):
            F[:, k - 1] = (2 * t * F[:, k] + np.exp(-t)) / (2 * k - 1)
        _TABLE.append(torch.tensor(F, device="cuda"))
    tab = _TABLE[0]
    far = T >= 48.0
    near = torch.where(far, 0.0, T)
    i = torch.round(near * 32.0).long()
    d = i.double() / 32.0 - near
    v = tab[i, m + 6]
    for k in range(5, -1, -1):
        v = v * (d / (k + 1)) + tab[i, m + k]
    rest = torch.where(far, T, 1.0)
    asym = 0.5 * math.sqrt(math.pi) * rest.rsqrt()
    for k in range(1, m + 1):
        asym = asym * ((2 * k - 1) / (2 * rest))
    F = [None] * m + [torch.where(far, asym, v)]
    e = torch.exp(-T)
    for k in range(m, 0, -1):
        F[k - 1] = (2 * T * F[k] + e) / (2 * k - 1)
    return F


def _R(L, p, P, C, zeta):
    """U R_tuv(rho, P - C) for t + u + v <= L, pairs along the first dimension and points along the second."""
    z2 = (zeta * zeta)[None, :]
    rho = p[:, None] * z2 / (p[:, None] + z2)
    U = torch.sqrt(z2 / (p[:, None] + z2))
    X = [P[:, d, None] - C[None, :, d] for d in range(3)]
    F = _boys(L, rho * (X[0] * X[0] + X[1] * X[1] + X[2] * X[2]))
    have, f = {}, U
    for n in range(L + 1):
        have[n] = f * F[n]
        f = f * (-2.0 * rho)
    level = {(0, 0, 0): have[L]}
    for n in range(L - 1, -1, -1):
        new = {(0, 0, 0): have[n]}
        for h in _herm(L - n)[1:]:
            d = 0 if h[0] else 1 if h[1] else 2
            one = tuple(x - (k == d) for k, x in enumerate(h))
            new[h] = X[d] * level[one]
            if h[d] > 1:
                two = tuple(x - 2 * (k == d) for k, x in enumerate(h))
                new[h] = new[h] + (h[d] - 1) * level[two]
        level = new
    return level


# -- exact values ------------------------------------------------------------------------------------------------------
def _surface(mol, xyz):
    """Points (in the library's order), exponents, switching factors, atoms."""
    i = np.arange(NPTS)
    z = 1.0 - (2.0 * i + 1.0) / NPTS
    phi = i * (math.pi * (3.0 - math.sqrt(5.0)))
    s = np.sqrt(1.0 - z * z)
    u = torch.tensor(np.stack([s * np.cos(phi), s * np.sin(phi), z], 1), device="cuda")
    R = torch.tensor(mol.radius, device="cuda")
    C = (xyz[:, None, :] + R[:, None, None] * u[None]).reshape(-1, 3)
    atom = torch.arange(mol.natom, device="cuda").repeat_interleave(NPTS)
    zeta = (ZETA / (R * math.sqrt(4 * math.pi / NPTS)))[atom]
    d = (C[:, None, :] - xyz[None]).square().sum(-1).sqrt()
    f = 0.5 * (torch.erfc(zeta[:, None] * (R[None] - d)) + torch.erfc(zeta[:, None] * (R[None] + d)))
    S = torch.where(atom[:, None] == torch.arange(mol.natom, device="cuda")[None], 1.0, f).prod(1)
    keep = torch.nonzero(S.detach() >= DROP)[:, 0]
    keep = keep[torch.argsort(zeta[keep], stable=True)]
    return C[keep], zeta[keep], S[keep], atom[keep]


def _A(C, zeta, S, rows=slice(None)):
    r = (C[rows][:, None, :] - C[None]).square().sum(-1)
    same = r == 0
    r = torch.where(same, 1.0, r).sqrt()
    zp = zeta[rows][:, None] * zeta[None] / torch.sqrt(zeta[rows][:, None] ** 2 + zeta[None] ** 2)
    return torch.where(same, (zeta * math.sqrt(2 / math.pi) / S)[rows][:, None].expand_as(r), torch.erf(zp * r) / r)


def _Bz(mol, xyz, C, zeta):
    d = (C[:, None, :] - xyz[None]).square().sum(-1).sqrt()
    return (torch.tensor(mol.Z, device="cuda")[None] * torch.erf(zeta[:, None] * d) / d).sum(1)


def _integrals(basis, xyz, P, C, zeta, q=None, dF=False, gradient=False):
    """c, and for charges q the Fock correction; or (gradient) the derivative of c.q at fixed P and q with respect to xyz
    (through the orbitals) and to the points."""
    prims = _prims(basis)
    n, M = basis.nbf, len(C)
    c = torch.zeros(M, dtype=torch.float64, device="cuda")
    out = torch.zeros(n * n, dtype=torch.float64, device="cuda") if dF else None
    gx, gC = torch.zeros_like(xyz), torch.zeros_like(C)
    for la, lb, i, j, w in _pairs(prims, xyz, 1e-15, max(1, 8_000_000 // M)):
        L = la + lb
        x = xyz.clone().requires_grad_(gradient)
        p, Pc, K, E = _expansion(prims, x, la, lb, i, j)
        pre = -(2.0 * math.pi / p) * K
        if P is not None:
            D = {h: 0.0 for h in _herm(L)}
            for a, b, f, row, col in _blocks(prims, la, lb, i, j):
                m = f * pre * torch.where(w > 1, P[row, col] + P[col, row], P[row, col])
                for h in D:
                    e = _product(E, a, b, h)
                    D[h] = D[h] if e is None else D[h] + m * e
        with torch.no_grad():
            R = _R(L + (1 if gradient else 0), p, Pc, C, zeta)
            W = {h: v @ q for h, v in R.items()} if q is not None else None
            if P is not None and not gradient:
                for h in D:
                    c += D[h] @ R[h]
            if dF:
                for a, b, f, row, col in _blocks(prims, la, lb, i, j):
                    v = 0.0
                    for h in _herm(L):
                        e = _product(E, a, b, h)
                        v = v if e is None else v + e * W[h]
                    v = f * pre * v
                    out.index_add_(0, row * n + col, torch.where((w > 1) if la == lb else (w > 0), v, 0.5 * v))
            if gradient:
                up = [{h: tuple(v + (k == d) for k, v in enumerate(h)) for h in D} for d in range(3)]
                gP = torch.stack([sum(D[h] * W[up[d][h]] for h in D) for d in range(3)], 1)
                for d in range(3):
                    for h in D:
                        gC[:, d] -= q * (D[h] @ R[up[d][h]])
        if gradient:
            terms = [(D[h], W[h]) for h in D if isinstance(D[h], torch.Tensor) and D[h].requires_grad]
            if Pc.requires_grad:
                terms.append((Pc, gP))
            gx += torch.autograd.grad([t[0] for t in terms], x, [t[1] for t in terms])[0]
        del R
    if dF:
        out = out.view(n, n)
        out = out + out.T
    return c, out, gx, gC


def _gradient(mol, basis, P, q):
    """Derivative of the energy at fixed P and q."""
    x = torch.tensor(mol.xyz, device="cuda", requires_grad=True)
    C, zeta, S, atom = _surface(mol, x)
    e = (_Bz(mol, x, C, zeta) * q).sum()
    g = torch.autograd.grad(e, x, retain_graph=True)[0]
    for k in range(0, len(C), 2048):
        r = slice(k, min(k + 2048, len(C)))
        e = (q[r] * (_A(C, zeta, S, r) @ q)).sum() / (2.0 * F_EPS)
        g = g + torch.autograd.grad(e, x, retain_graph=True)[0]
    _, _, gx, gC = _integrals(basis, x.detach(), P, C.detach(), zeta.detach(), q=q, gradient=True)
    return g + gx + torch.zeros_like(gx).index_add_(0, atom, gC)


def exact(case, seed):
    if case["call"] == "batch" or case["natom"] > 300 or case["call"] in ("opt", "gradient") and case["natom"] > 120:
        return None
    s = _inputs(case, seed)
    mol, basis, P = s["mol"], s["basis"], s["Pd"]
    xyz = torch.tensor(mol.xyz, device="cuda")
    if case["call"] in ("fock", "gradient"):      # the charges are an input of these
        q = prepare(case, seed)["q"]
        q = q if isinstance(q, torch.Tensor) else torch.tensor(q, device="cuda")
        if case["call"] == "gradient":
            return {"g": _gradient(mol, basis, P, q)}
        C, zeta, _, _ = _surface(mol, xyz)
        return {"dF": _integrals(basis, xyz, None, C, zeta, q=q, dF=True)[1]}
    C, zeta, S, _ = _surface(mol, xyz)
    c = _integrals(basis, xyz, P, C, zeta)[0]
    if case["call"] == "esp":
        return {"c": c}
    A, Bz = _A(C, zeta, S), _Bz(mol, xyz, C, zeta)
    q = torch.cholesky_solve((-F_EPS * (Bz + c))[:, None], torch.linalg.cholesky(A))[:, 0]
    if case["call"] == "solve":
        return {"q": q}
    got = {"c": c, "q": q, "dF": _integrals(basis, xyz, None, C, zeta, q=q, dF=True)[1],
           "E": float((Bz + c) @ q + q @ (A @ q) / (2.0 * F_EPS))}
    if case["call"] == "opt":
        got["g"] = _gradient(mol, basis, P, q)
    return got


# -- the calls ---------------------------------------------------------------------------------------------------------
def _inputs(case, seed):
    mol, basis = _molecule(case["natom"], case["d_shells"], seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nocc = min(5 if case["natom"] == 3 else 2 * case["natom"], basis.nbf)
    P = _density(basis, torch.tensor(mol.xyz, device="cuda"), nocc, gen)
    return {"mol": mol, "basis": basis, "Pd": P, "P": P.cpu().numpy() if case["host"] else P}


def prepare(case, seed):
    if case["call"] == "batch":
        batch = pcm.Batch(case["nmol"], precision=case["precision"])
        sizes = np.random.default_rng([case["natom"], case["nmol"]]).uniform(0.8, 1.2, case["nmol"])
        Ps = []
        for k in range(case["nmol"]):
            natom = max(4, int(case["natom"] * sizes[k]))
            s = _inputs(dict(case, natom=natom), 1000 * seed + k)
            batch.set_molecule(k, s["mol"], s["basis"])
            Ps.append(s["Pd"])
        torch.cuda.synchronize()
        return {"case": case, "batch": batch, "Ps": Ps}
    s = _inputs(case, seed)
    s["case"] = case
    s["ctx"] = ctx = pcm.Context(precision=case["precision"])
    torch.cuda.synchronize()
    if case["call"] not in ("step", "opt"):       # an SCF's context stands at its geometry
        ctx.setup(s["mol"], s["basis"])
    if case["call"] in ("solve", "fock", "gradient"):
        ctx.esp(s["P"])
        if case["call"] != "solve":
            s["q"], _ = ctx.solve(prev_diis_error=case["diis"], like=s["P"])
    return s


def run(s):
    call, diis = s["case"]["call"], s["case"]["diis"]
    if call == "batch":
        E, q, dF = s["batch"].run(s["Ps"], pcm.cg_threshold(prev_diis_error=diis), want_q=True, want_dF=True)
        return {"E": E, "q": q, "dF": dF}
    ctx, P = s["ctx"], s["P"]
    if call == "esp":
        return {"c": ctx.esp(P)}
    if call == "solve":
        return {"q": ctx.solve(prev_diis_error=diis, like=P)[0]}
    if call == "fock":
        return {"dF": ctx.fock(s["q"])}
    if call == "gradient":
        return {"g": ctx.gradient(s["q"], P)}
    if call in ("step", "opt"):
        ctx.setup(s["mol"], s["basis"])
    c = ctx.esp(P)
    q, _ = ctx.solve(prev_diis_error=diis, like=P)
    got = {"c": c, "q": q, "dF": ctx.fock(q), "E": ctx.energy(q)}
    if call == "opt":
        got["g"] = ctx.gradient(q, P)
    return got


def work(case):
    """Bytes: the density and the Fock correction, each once, and the vectors over the points.  Operations: two for each
    element of the operator that a solve cannot do without, and for the integrals two for each shell pair of atoms near
    enough to overlap and each of its basis-function pairs' Hermite terms (the pairs' own set-up; the contraction over the
    points can be shared between pairs)."""
    n = case["natom"]
    per = 8.6 if case["d_shells"] else 5.6
    nbf, M = per * n, (84.0 if n == 3 else 46.0) * n
    npair = min(0.5 * n * n, 60.0 * n)
    call = case["call"]
    bytes_ = 8.0 * M
    flops = 0.0
    if call != "solve":
        bytes_ += 8.0 * nbf * nbf * (2 if call in ("step", "scf", "opt", "batch") else 1)
        flops += npair * per * per * 100.0
    if call not in ("esp", "fock"):
        flops += 2.0 * M * M
    if call in ("step", "scf", "opt", "batch"):
        flops += npair * per * per * 100.0
    k = max(1, case["nmol"])
    return {"bytes": k * bytes_, "flops": k * flops}
