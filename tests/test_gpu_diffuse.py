"""PCM_FP64 Fock correction with the cells' expansions on and functions so diffuse
(exponent 2^-16) that their near form is far below the far form at every distance in the
molecule: their elements against the oracle, which evaluates them directly."""
import numpy as np
import pytest

import _expansions
import oracle
import workloads
from _parity import FP64, check

pytestmark = pytest.mark.gpu


def test_diffuse_functions():
    import paper_1505_07851_gb300 as pcm
    w = workloads.small_cluster(130, seed=91, d_shells=True)
    b = w.basis
    atoms = np.array([3, 50, 90, 129], np.int32)
    b.shell_atom = np.concatenate([b.shell_atom, np.repeat(atoms, 2)])
    b.shell_l = np.concatenate([b.shell_l, np.tile(np.array([1, 2], np.int32), 4)])
    b.shell_nprim = np.concatenate([b.shell_nprim, np.ones(8, np.int32)])
    b.exps = np.concatenate([b.exps, np.full(8, 2.0 ** -16)])
    b.coefs = np.concatenate([b.coefs, np.ones(8)])
    with pcm.Context(precision="fp64") as ctx:
        M, nbf = ctx.setup(w.mol, b)
        assert _expansions.on(ctx.stats(), True)
        q = np.random.default_rng(11).uniform(0.0, 1.0, M)
        dF = ctx.fock(q)
        xyzzs = ctx.get_surface()[0]
    eb = oracle.ExpandedBasis(b, w.mol.xyz)
    own = np.flatnonzero(eb.exps[eb.sh_off] == 2.0 ** -16)
    pairs = [(i, j) for i in own for j in own if i <= j]
    blocks = oracle.fock_blocks(eb, q, xyzzs[:, :3], xyzzs[:, 3], pairs)
    for (i, j), ref in zip(pairs, blocks):
        fi, fj = eb.sh_bf[i], eb.sh_bf[j]
        check(dF[fi:fi + ref.shape[0], fj:fj + ref.shape[1]], ref, FP64, what="block %d %d" % (i, j))
