"""Primitive pairs kept by the Schwarz screening against a NumPy evaluation of the
bound |c_a c_b| max (ab|ab)^(1/2) from the diagonal two-electron integrals: s, p
and d shells, exponents from 1e-3 to 1e7, near and far centres, cutoffs between
all and few pairs.  The count is exact in FP64 but for pairs whose bound is
within 1e-9 of the cutoff (none here), in PCM_MIXED, whose bound is FP32, but for
those within 1e-4 of it."""
import numpy as np
import pytest

import oracle
import workloads
from oracle.pcm import cart_exponents

pytestmark = pytest.mark.gpu


def _dfact(n):
    r = 1.0
    for k in range(n, 1, -2):
        r *= k
    return r


def _hermite(la, lb, pa, pb, h):
    """E[i, j, t] of x_A^i x_B^j without the exponential prefactor; h = 1 / 2p."""
    E = np.zeros((la + 1, lb + 1, la + lb + 3) + pa.shape)
    E[0, 0, 0] = 1.0
    t = np.arange(1, la + lb + 2).reshape(-1, *([1] * pa.ndim))

    def up(e, x):
        out = np.zeros_like(e)
        out[0] = x * e[0] + e[1]
        out[1:-1] = h * e[:-2] + x * e[1:-1] + (t + 1) * e[2:]
        return out

    for i in range(la + 1):
        if i:
            E[i, 0] = up(E[i - 1, 0], pa)
        for j in range(1, lb + 1):
            E[i, j] = up(E[i, j - 1], pb)
    return E


def schwarz_bounds(eb):
    """Bounds of all primitive pairs (each unordered pair once)."""
    out = []
    for A in range(eb.nshell):
        for B in range(A + 1):
            la, lb = int(eb.sh_l[A]), int(eb.sh_l[B])
            oa, ob = eb.sh_off[A], eb.sh_off[B]
            a = eb.exps[oa:oa + eb.sh_nprim[A], None]
            b = eb.exps[None, ob:ob + eb.sh_nprim[B]]
            ca, cb = eb.coefs[oa:oa + eb.sh_nprim[A], None], eb.coefs[None, ob:ob + eb.sh_nprim[B]]
            RA, RB = eb.xyz[eb.sh_atom[A]], eb.xyz[eb.sh_atom[B]]
            p = a + b
            P = [(a * RA[d] + b * RB[d]) / p for d in range(3)]
            K2 = np.exp(-2.0 * a * b / p * ((RA - RB) ** 2).sum())
            E = [_hermite(la, lb, P[d] - RA[d], P[d] - RB[d], 0.5 / p) for d in range(3)]
            LL = la + lb
            best = np.zeros(p.shape)
            for ea in cart_exponents(la):
                for e_b in cart_exponents(lb):
                    G = []
                    for d in range(3):
                        e = E[d][ea[d], e_b[d]]
                        g = np.zeros((2 * LL + 1,) + p.shape)
                        for t in range(LL + 1):
                            for u in range(LL + 1):
                                g[t + u] += e[t] * e[u] * (-1.0) ** u
                        G.append(g)
                    s = 0.0
                    for T in range(0, 2 * LL + 1, 2):
                        for U in range(0, 2 * LL + 1 - T, 2):
                            for V in range(0, 2 * LL + 1 - T - U, 2):
                                n = (T + U + V) // 2
                                s = s + (G[0][T] * G[1][U] * G[2][V] * (-p) ** n * _dfact(T - 1) * _dfact(U - 1)
                                         * _dfact(V - 1) / (2 * n + 1))
                    f = np.prod([_dfact(2 * l - 1) for l in (la, lb)])
                    f /= np.prod([_dfact(2 * x - 1) for x in (*ea, *e_b)])
                    best = np.maximum(best, f * np.abs(s))
            eri = 2.0 * np.pi ** 2.5 / (p * p * np.sqrt(2.0 * p)) * K2 * best
            na = ca * (2 * a / np.pi) ** 0.75 * (4 * a) ** (0.5 * la) / np.sqrt(_dfact(2 * la - 1))
            nb = cb * (2 * b / np.pi) ** 0.75 * (4 * b) ** (0.5 * lb) / np.sqrt(_dfact(2 * lb - 1))
            Q = np.abs(na * nb) * np.sqrt(eri)
            out.append(Q[np.triu_indices(Q.shape[0])] if A == B else Q.ravel())
    return np.concatenate(out)


def _workload(name):
    w = workloads.small_cluster(9, seed=41, d_shells=True)
    rng = np.random.default_rng(42)
    if name != "plain":
        w.basis.exps = 10.0 ** rng.uniform(-3.0, 7.0, len(w.basis.exps))
        w.basis.coefs = w.basis.coefs * 10.0 ** rng.uniform(-6.0, 2.0, len(w.basis.coefs))
    if name == "far":
        w.mol.xyz = w.mol.xyz * 6.0 + np.array([300.0, -200.0, 100.0])
    return w


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["plain", "wide", "far"])
def test_pairs_kept(name, precision):
    import paper_1505_07851_gb300 as pcm
    w = _workload(name)
    Q = schwarz_bounds(oracle.ExpandedBasis(w.basis, w.mol.xyz))
    band = 1e-9 if precision == "fp64" else 1e-4
    for thresh in (0.0, 1e-30, 1e-12, 1e-6, 1e-2):
        with pcm.Context(precision=precision, schwarz=thresh) as ctx:
            ctx.setup(w.mol, w.basis)
            st = ctx.stats()
        assert st["pairs_candidate"] == len(Q)
        if thresh == 0.0:
            assert st["pairs_kept"] == len(Q)
        else:
            lo, hi = (Q >= thresh * (1 + band)).sum(), (Q >= thresh * (1 - band)).sum()
            assert lo <= st["pairs_kept"] <= hi, (thresh, lo, hi)
