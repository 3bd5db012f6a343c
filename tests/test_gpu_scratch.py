"""Device memory that a PCM_FP64 context takes for the Fock correction and the gradient
of 130 atoms with d shells, with the cells' expansions on: partial sums and raw moments
are bounded at 128 MB each, everything else (pair data, tables of coefficients, sums per
point) is a few megabytes each: 512 MB.  Measured on a second context: the first one's
launches make the driver reserve what it keeps for the process (local memory of kernels
with a stack)."""
import numpy as np
import pytest

import _expansions
import workloads

pytestmark = pytest.mark.gpu


def _memory_taken(w):
    import torch
    import paper_1505_07851_gb300 as pcm
    with pcm.Context(precision="fp64") as ctx:
        M, _ = ctx.setup(w.mol, w.basis)
        assert _expansions.on(ctx.stats(), True)
        q = np.full(M, 1e-2)
        ctx.apply_a(q)                     # the operator (A) is not scratch
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx.fock(q)
        ctx.gradient(q, w.P, terms="C")
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0]


def test_scratch_is_bounded():
    w = workloads.small_cluster(130, seed=97, d_shells=True)
    _memory_taken(w)
    took = _memory_taken(w)
    assert took <= 512 << 20, took
