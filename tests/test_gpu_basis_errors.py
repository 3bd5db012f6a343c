"""A basis that cannot be set: one that is refused leaves the context with its own, one
that runs out of memory half-way leaves it without any (and later calls are not disturbed
by the failed allocation)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_failed_set_basis(precision):
    import paper_1505_07851_gb300 as pcm
    w = workloads.small_cluster(6, seed=98, d_shells=True)
    b = w.basis
    shells = (b.shell_atom, b.shell_l, b.shell_nprim, b.exps, b.coefs)
    with pcm.Context(precision=precision) as ctx:
        M, _ = ctx.setup(w.mol, b)
        q = np.full(M, 1e-2)
        dF, g = ctx.fock(q), ctx.gradient(q, w.P, terms="C")
    with pcm.Context(precision=precision) as ctx:
        ctx.setup(w.mol, b)
        with pytest.raises(pcm.PCMError) as e:
            ctx.set_basis([0, 1], [0, 3], [1, 1], [1.0, 1.0], [1.0, 1.0])
        assert e.value.status == pcm.PCM_ERR_UNSUPPORTED
        assert np.array_equal(ctx.fock(q), dF) and np.array_equal(ctx.gradient(q, w.P, terms="C"), g)
        n = 1000000                                # 5e11 candidate pairs: their flags fit no device
        with pytest.raises(pcm.PCMError) as e:
            ctx.set_basis([0], [0], [n], np.ones(n), np.ones(n))
        assert e.value.status == pcm.PCM_ERR_OOM
        with pytest.raises(pcm.PCMError) as e:
            ctx.fock(q)
        assert e.value.status == pcm.PCM_ERR_ARG
        ctx.set_basis(*shells)
        assert np.array_equal(ctx.fock(q), dF) and np.array_equal(ctx.gradient(q, w.P, terms="C"), g)
