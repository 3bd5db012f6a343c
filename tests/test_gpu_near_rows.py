"""Surfaces and the matrix-free operator's near rows where their FP32 tests can go
wrong: fewer points than a warp, ragged last blocks, atoms with their own radii and
point spacing, scattered atoms, and molecules far from the origin (coarser FP32
coordinates).  The kept points are the oracle's; the products of a positive vector
hold 1e-11 (accurate) and 1e-6 relative (FP32), the latter plus the rounding of the
coordinates: 2 sqrt(3) 2^-24 |x| in a distance of 2 bohr or more."""
import numpy as np
import pytest

import oracle
import workloads
from _parity import check

pytestmark = pytest.mark.gpu


def _molecule(name):
    if name == "atom":
        return np.zeros((1, 3)), np.array([8.0]), np.array([3.2]), 19
    w = workloads.small_cluster(23, seed=51)
    xyz, Z, radius, n = w.mol.xyz.copy(), w.mol.Z, w.mol.radius, 110
    if name == "radii":
        radius, n = radius * np.linspace(0.7, 1.4, len(Z)), 37
    if name == "distant":
        xyz += np.array([900.0, -700.0, 400.0])
    if name == "scattered":
        xyz *= 8.0
    return xyz, Z, radius, n


@pytest.mark.parametrize("name", ["atom", "compact", "radii", "distant", "scattered"])
def test_surface_and_near_rows(name):
    import paper_1505_07851_gb300 as pcm
    xyz, Z, radius, n = _molecule(name)
    s = oracle.surface(xyz, radius, n=n)
    with pcm.Context(precision="mixed", operator="free") as ctx:
        M = ctx.build_surface(xyz, Z, radius, n)
        xyzzs, idx = ctx.get_surface()
        x = np.random.default_rng(6).uniform(0.0, 1.0, M)
        y, y32 = np.array(ctx.apply_a(x)), np.array(ctx.apply_a(x, fp32=True))
    assert sorted(idx) == sorted(s["index"])
    ref = oracle.a_matrix({"r": xyzzs[:, :3], "zeta": xyzzs[:, 3], "S": xyzzs[:, 4]}) @ x
    check(y, ref, (1e-11, 0.0), what="accurate product")
    check(y32, ref, (1e-6 + 1.04e-7 * np.abs(xyzzs[:, :3]).max(), 0.0), what="FP32 product")
