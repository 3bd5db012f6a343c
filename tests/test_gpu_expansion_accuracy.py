"""PCM_FP64 with the cells' expansions on: single elements against closed forms.

One-centre products of tight functions see every point in the far form, so their
elements are derivatives of 1/R: for exponents a = p/2 a power of two at coordinates
that are multiples of 2^-10 (the pair's centre is the atom to the last bit),
  <px|1/R|py> = 3XY / (2p R^5),
  <dxx|1/R|dxy> = sqrt(3) 4p^2/3 ((105 X^3 Y / R^9 - 45 X Y / R^7) / (2p)^4 + 9XY / (2p)^3 R^5),
pure second and fourth derivatives, which no lower term hides.  Single charges show the
truncation of one expansion, charges of one sign that of all.  Bars: an expansion's sums
round to 2.5e-15 of the derivative's norm in the worst case (a pair at the rim of its
cell, the closest points admitted; evaluated in NumPy at orders 24 and 30), the
normalisation and the contraction to another ten roundings: 1e-14 of the sum of the norms.
The gradient's centre parts are differences of terms of the size of 1/R^2, those of the
points pure third derivatives: 2e-14 of the sums of those."""
import numpy as np
import pytest

import _expansions
import workloads

pytestmark = pytest.mark.gpu

A = 64.0
PP = 2.0 * A


def _workload():
    w = workloads.small_cluster(130, seed=81, d_shells=True)
    w.mol.xyz = np.round(w.mol.xyz * 1024.0) / 1024.0
    b = w.basis
    # atoms with every point beyond T = 60
    atoms = np.array([0, 8, 12, 15, 19, 22, 26, 30, 36, 40, 47, 52, 57, 65, 79, 83, 87, 95, 103, 121], np.int32)
    first = b.nbf + 9 * np.arange(len(atoms))          # a p and a d shell each, after the molecule's own
    b.shell_atom = np.concatenate([b.shell_atom, np.repeat(atoms, 2)])
    b.shell_l = np.concatenate([b.shell_l, np.tile(np.array([1, 2], np.int32), len(atoms))])
    b.shell_nprim = np.concatenate([b.shell_nprim, np.ones(2 * len(atoms), np.int32)])
    b.exps = np.concatenate([b.exps, np.full(2 * len(atoms), A)])
    b.coefs = np.concatenate([b.coefs, np.ones(2 * len(atoms))])
    return w, atoms, first


def _context(w):
    import paper_1505_07851_gb300 as pcm
    ctx = pcm.Context(precision="fp64")
    ctx.setup(w.mol, w.basis)
    assert _expansions.on(ctx.stats(), True)
    return ctx


def _charges(kind, M, rng):
    if kind == "one sign":
        return [np.full(M, 1e-2)]
    out = []
    for k in rng.choice(M, 16, replace=False):
        q = np.zeros(M)
        q[k] = 1.0
        out.append(q)
    return out


@pytest.mark.parametrize("kind", ["single", "one sign"])
def test_elements(kind):
    w, atoms, first = _workload()
    rng = np.random.default_rng(9)
    worst = {"p": 0.0, "d": 0.0}
    with _context(w) as ctx:
        pts = ctx.get_surface()[0].astype(np.longdouble)
        for q in _charges(kind, len(pts), rng):
            dF = ctx.fock(q)
            on = np.flatnonzero(q)
            for a, f in zip(atoms, first):
                X, Y, Z = (w.mol.xyz[a].astype(np.longdouble) - pts[on, :3]).T
                R = np.sqrt(X * X + Y * Y + Z * Z)
                rho = PP * pts[on, 3] ** 2 / (PP + pts[on, 3] ** 2)
                assert (rho * R * R).min() > 60.0
                qk = q[on].astype(np.longdouble)
                for i, j, u, v in ((0, 1, X, Y), (0, 2, X, Z), (1, 2, Y, Z)):
                    ref = -(qk * 3 * u * v / (2 * PP * R ** 5)).sum()
                    scale = (abs(qk) * 3 / (2 * PP * R ** 3)).sum()
                    worst["p"] = max(worst["p"], float(abs(dF[f + i, f + j] - ref) / scale))
                c = np.sqrt(np.longdouble(3)) * 4 * PP ** 2 / 3
                ref = -c * (qk * ((105 * X ** 3 * Y / R ** 9 - 45 * X * Y / R ** 7) / (2 * PP) ** 4
                                  + 9 * X * Y / ((2 * PP) ** 3 * R ** 5))).sum()
                scale = c * (abs(qk) * (105 / ((2 * PP) ** 4 * R ** 5) + 9 / ((2 * PP) ** 3 * R ** 3))).sum()
                worst["d"] = max(worst["d"], float(abs(dF[f + 3, f + 4] - ref) / scale))
    assert worst["p"] <= 1e-14 and worst["d"] <= 1e-14, worst


def test_gradient_of_single_charges():
    w, atoms, first = _workload()
    rng = np.random.default_rng(10)
    n = w.basis.nbf
    P = np.zeros((n, n))
    d = rng.uniform(0.5, 1.0, len(atoms)) * rng.choice([-1.0, 1.0], len(atoms))
    P[first, first + 1] = P[first + 1, first] = d          # the px py elements
    worst = {"centre": 0.0, "point": 0.0}
    with _context(w) as ctx:
        pts, idx = ctx.get_surface()
        owner = np.asarray(idx) // 110
        for k in rng.choice(np.flatnonzero(~np.isin(owner, atoms)), 12, replace=False):
            q = np.zeros(len(pts))
            q[k] = 1.0
            g = ctx.gradient(q, P, terms="C")
            V = w.mol.xyz[atoms].astype(np.longdouble) - pts[k, :3].astype(np.longdouble)
            X, Y, Z = V.T
            R = np.sqrt((V * V).sum(1))
            # derivatives of 3XY / R^5 with respect to the centre
            ref = np.stack([3 * Y / R ** 5 - 15 * X * X * Y / R ** 7, 3 * X / R ** 5 - 15 * X * Y * Y / R ** 7,
                            -15 * X * Y * Z / R ** 7], 1) * (-2 * d / (2 * PP))[:, None]
            err = np.abs(g[atoms] - ref) / (np.abs(2 * d) / R ** 2)[:, None]
            worst["centre"] = max(worst["centre"], float(err.max()))
            scale = (np.abs(2 * d) * 15 / (2 * PP * R ** 4)).sum()
            worst["point"] = max(worst["point"], float(np.abs(g[owner[k]] + ref.sum(0)).max() / scale))
    assert worst["centre"] <= 2e-14 and worst["point"] <= 2e-14, worst
