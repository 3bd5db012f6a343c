"""PCM_FP64 Fock correction and gradient of molecules whose parts lie so far apart that
their squared distances leave FP32's range (2^67, 2^80 bohr): the oracle's values for the
part at the origin (the distant atom's own pair centres are off by FP64's spacing there)."""
import numpy as np
import pytest

import oracle
import workloads
from _parity import FP64, check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("apart", [2.0 ** 40, 2.0 ** 67, 2.0 ** 80])
def test_parts_far_apart(apart):
    import paper_1505_07851_gb300 as pcm
    w = workloads.small_cluster(6, seed=61, d_shells=True)
    w.mol.xyz[-1] = [apart, 0.0, -apart]
    with pcm.Context(precision="fp64", schwarz=0.0) as ctx:
        M, nbf = ctx.setup(w.mol, w.basis)
        q = np.random.default_rng(7).uniform(-1.0, 0.3, M) * 1e-2
        dF = ctx.fock(q)
        g = ctx.gradient(q, w.P, terms="C")
        xyzzs, idx = ctx.get_surface()
    s = oracle.surface(w.mol.xyz, w.mol.radius)
    pos = {int(k): i for i, k in enumerate(s["index"])}
    q_o = np.empty(M)
    q_o[[pos[int(k)] for k in idx]] = q
    eb = oracle.ExpandedBasis(w.basis, w.mol.xyz)
    n = eb.sh_bf[eb.sh_atom == w.mol.natom - 1].min()
    check(dF[:n, :n], oracle.fock(eb, q_o, s["r"], s["zeta"])[:n, :n], FP64, what="dF")
    check(g[:-1], oracle.gradient_c(eb, w.P, q_o, s)[:-1], FP64, what="gradient")
