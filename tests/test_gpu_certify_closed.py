"""Certificates of vectors that hold anything on closed faces away from the cavity: rho and the
Rayleigh quotient are of the open faces, and closed faces that share no edge or cell with one
have no part in them."""
import numpy as np
import pytest

import workloads as W
from oracle import geometry, operators

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(20, 12, 14), (38, 10, 9)])
def test_closed_faces_out_of_reach(n, dm, ctx):
    g = W.Grid(*n, 0.1, 0.1, 0.1, (0.0, 0.0, 0.0))
    mid = [0.05 * v for v in n]
    w = W.Workload("w", g, W.ellipsoid_phi(g, mid, [0.6 * v for v in mid]), 2.0, 1, 0)
    geom = dm.Geometry.from_workload(ctx, w)
    ops = operators.DMOperators(w.grid, geometry.fractions(w.phi))
    nx, ny, nz = n
    # nodes within two of an open face's
    dims = [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)]
    off = np.concatenate([[0], np.cumsum([int(np.prod(d)) for d in dims])])
    near = np.zeros((nz + 5, ny + 5, nx + 5), bool)
    for c, d in enumerate(dims):
        k, j, i = np.nonzero(ops.open[off[c]:off[c + 1]].reshape(d))
        for dk in range(5):
            for dj in range(5):
                for di in range(5):
                    near[k + dk, j + dj, i + di] = True
    far = np.concatenate([~near[2:2 + d[0], 2:2 + d[1], 2:2 + d[2]].ravel() for d in dims])
    assert far.sum() > 10 and not ops.open[far].any()
    rng = np.random.default_rng(1)
    B = rng.standard_normal((2, ops.a.size)) * ops.open
    k2 = [4.0, 9.0]
    want = dm.certify(ctx, geom, k2, B)
    for bad in (np.nan, np.inf, 1e300):
        C = B.copy()
        C[:, far] = bad
        got = dm.certify(ctx, geom, k2, C)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[2], want[2]), bad
