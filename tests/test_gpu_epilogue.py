"""The Fock epilogue's two layouts (eight lanes, or a thread, per shell pair, by the
elements of a class and its primitive pairs per shell pair) in every class and both
precisions against the oracle: few shells of one, two and four primitives (all eight
lanes), and enough shells of one primitive that the d classes take the other layout."""
import numpy as np
import pytest

import oracle
import workloads
from _parity import FP64, MIXED, check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,bars", [("fp64", FP64), ("mixed", MIXED)])
@pytest.mark.parametrize("natom,nprim", [(7, 1), (7, 2), (7, 4), (130, 1)])
def test_contractions(natom, nprim, precision, bars):
    import paper_1505_07851_gb300 as pcm
    w = workloads.small_cluster(natom, seed=95)
    rng = np.random.default_rng(12)
    n = 3 * natom
    b = workloads.Basis(np.repeat(np.arange(natom, dtype=np.int32), 3), np.tile(np.array([0, 1, 2], np.int32), natom),
                        np.full(n, nprim, np.int32), np.exp(rng.uniform(-1.5, 3.0, n * nprim)),
                        rng.uniform(0.1, 1.0, n * nprim))
    with pcm.Context(precision=precision, schwarz=0.0) as ctx:
        M, nbf = ctx.setup(w.mol, b)
        q = rng.uniform(-1.0, 0.3, M) * 1e-2
        dF = ctx.fock(q)
        xyzzs = ctx.get_surface()[0]
    eb = oracle.ExpandedBasis(b, w.mol.xyz)
    pairs = [(i, j) for i in range(n) for j in range(i, n)]
    if natom > 10:
        pairs = [pairs[k] for k in rng.choice(len(pairs), 60, replace=False)] + [(i, i) for i in range(0, n, 16)]
    blocks = oracle.fock_blocks(eb, q, xyzzs[:, :3], xyzzs[:, 3], pairs)
    got, ref = [], []
    for (i, j), blk in zip(pairs, blocks):
        fi, fj = eb.sh_bf[i], eb.sh_bf[j]
        got += [dF[fi:fi + blk.shape[0], fj:fj + blk.shape[1]].ravel(), dF[fj:fj + blk.shape[1], fi:fi + blk.shape[0]].T.ravel()]
        ref += [blk.ravel(), blk.ravel()]
    check(np.concatenate(got), np.concatenate(ref), bars, scale=float(np.max(np.abs(dF))), what="dF")
