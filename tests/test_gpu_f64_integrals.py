"""PCM_FP64 Fock correction and gradient integrals against the oracle at the
sizes where their point tiles (32) and sorted pairs begin: surfaces below and
above the sorting thresholds (1024 points, 4096 pairs), ragged last tiles, more
exponent classes than are tabulated (16), and enough pairs (20000) for the
cells' multipole and local expansions, in a compact and in a stretched molecule
(more far tiles, higher orders).  FP64 bars of _parity."""
import numpy as np
import pytest

import oracle
import workloads
from _parity import FP64, check

pytestmark = pytest.mark.gpu


def _many_radii(natom, seed):
    """A cluster whose atoms all have their own cavity radius."""
    w = workloads.small_cluster(natom, seed=seed, d_shells=True)
    w.mol.radius = w.mol.radius * np.linspace(0.95, 1.05, natom)
    return w


def _stretched(natom, seed, d_shells):
    w = workloads.small_cluster(natom, seed=seed, d_shells=d_shells)
    half = np.arange(natom) >= natom // 2
    w.mol.xyz[half] += np.array([20.0, -9.0, 5.0])
    return w


CASES = {
    "cluster45_sp": lambda: workloads.small_cluster(45, seed=35),
    "stretched52_spd": lambda: _stretched(52, 36, True),
    "water": lambda: workloads.config(0),
    "cluster5_spd": lambda: workloads.small_cluster(5, seed=31, d_shells=True),
    "cluster20_spd": lambda: workloads.small_cluster(20, seed=32, d_shells=True),
    "cluster26_sp": lambda: workloads.small_cluster(26, seed=33),
    "radii17_spd": lambda: _many_radii(17, 34),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_fock_and_gradient_against_oracle(name):
    import paper_1505_07851_gb300 as pcm
    w = CASES[name]()
    rng = np.random.default_rng(5)
    with pcm.Context(precision="fp64", schwarz=0.0) as ctx:
        M, nbf = ctx.setup(w.mol, w.basis)
        q = rng.uniform(-1.0, 0.3, M) * 1e-2
        dF = ctx.fock(q)
        again = ctx.fock(q)
        g = ctx.gradient(q, w.P)
        xyzzs, idx = ctx.get_surface()
    assert np.array_equal(dF, again)
    s = oracle.surface(w.mol.xyz, w.mol.radius)
    pos = {int(k): i for i, k in enumerate(s["index"])}
    p = np.array([pos[int(k)] for k in idx])
    q_o = np.empty(M)
    q_o[p] = q
    eb = oracle.ExpandedBasis(w.basis, w.mol.xyz)
    check(dF, oracle.fock(eb, q_o, s["r"], s["zeta"]), FP64, what="dF")
    ref = oracle.gradient(eb, w.P, q_o, s, w.mol.xyz, w.mol.Z, w.mol.radius, oracle.f_factor())["total"]
    check(g, ref, FP64, what="gradient")
