"""PCM_FP64 Fock correction with the cells' expansions on (asserted by the library's
thresholds), against the oracle: a compact s/p and a compact s/p/d molecule, a stretched
one (more far tiles, higher orders), and one whose atoms all have their own radius (more
exponent classes than are tabulated).  Sampled shell blocks for all charges, FP64 bars of
_parity."""
import numpy as np
import pytest

import _expansions
import oracle
import workloads
from _parity import FP64, check

pytestmark = pytest.mark.gpu


def _molecule(name):
    d = name != "compact_sp"
    w = workloads.small_cluster(105 if not d else 130, seed=101, d_shells=d)
    if name == "stretched":
        w.mol.xyz[w.mol.natom // 2:] += np.array([24.0, -11.0, 6.0])
    if name == "radii":
        w.mol.radius = w.mol.radius * np.linspace(0.95, 1.05, w.mol.natom)
    return w, d


@pytest.mark.parametrize("name", ["compact_sp", "compact_spd", "stretched", "radii"])
def test_fock_against_oracle(name):
    import paper_1505_07851_gb300 as pcm
    w, d = _molecule(name)
    rng = np.random.default_rng(13)
    with pcm.Context(precision="fp64", schwarz=0.0) as ctx:
        M, nbf = ctx.setup(w.mol, w.basis)
        assert _expansions.on(ctx.stats(), d)
        q = rng.uniform(-1.0, 0.3, M) * 1e-2
        dF = ctx.fock(q)
        assert np.array_equal(dF, ctx.fock(q))
        xyzzs = ctx.get_surface()[0]
    if name == "radii":
        assert len(np.unique(xyzzs[:, 3])) > 16
    eb = oracle.ExpandedBasis(w.basis, w.mol.xyz)
    pairs = [tuple(sorted(rng.choice(eb.nshell, 2))) for _ in range(40)] + [(a, a) for a in range(0, eb.nshell, 20)]
    got, ref = [], []
    for (i, j), blk in zip(pairs, oracle.fock_blocks(eb, q, xyzzs[:, :3], xyzzs[:, 3], pairs)):
        fi, fj = eb.sh_bf[i], eb.sh_bf[j]
        got.append(dF[fi:fi + blk.shape[0], fj:fj + blk.shape[1]].ravel())
        ref.append(blk.ravel())
    check(np.concatenate(got), np.concatenate(ref), FP64, scale=float(np.max(np.abs(dF))), what="dF")
