"""PCM_FP64 Fock correction and gradient far from the origin, with the cells'
expansions on: the interactions' near and far forms are chosen in FP32, by coordinates
that count from the middle of the molecule, so a translation by 2^24 bohr (FP32 spacing
there: 2 bohr) changes nothing but the FP64 rounding of the points and centres.  That
rounding, 4e-9 bohr, reaches an element as up to sqrt(2p) and a gradient as up to 2p
sqrt(2p) times itself (p <= 40: 4e-8, 3e-6); the bars are 1e-5 and 1e-4 of the largest
element."""
import numpy as np
import pytest

import _expansions
import workloads
from _parity import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natom,d_shells", [(12, True), (130, True)])
def test_translation(natom, d_shells):
    import paper_1505_07851_gb300 as pcm
    w = workloads.small_cluster(natom, seed=71, d_shells=d_shells)
    w.basis.exps = np.minimum(w.basis.exps, 20.0)
    w.mol.xyz = np.round(w.mol.xyz * 1024.0) / 1024.0
    got = []
    for shift in ([0.0, 0.0, 0.0], [2.0 ** 24, -2.0 ** 24, 2.0 ** 23]):
        with pcm.Context(precision="fp64") as ctx:
            M = ctx.build_surface(w.mol.xyz + np.array(shift), w.mol.Z, w.mol.radius)
            b = w.basis
            ctx.set_basis(b.shell_atom, b.shell_l, b.shell_nprim, b.exps, b.coefs)
            assert natom < 100 or _expansions.on(ctx.stats(), d_shells)
            q = np.random.default_rng(8).uniform(-1.0, 0.3, M) * 1e-2
            got.append((ctx.get_surface()[1], ctx.fock(q), ctx.gradient(q, w.P, terms="C")))
    assert np.array_equal(got[0][0], got[1][0])
    check(got[1][1], got[0][1], (0.0, 1e-5), what="dF")
    check(got[1][2], got[0][2], (0.0, 1e-4), what="gradient")
