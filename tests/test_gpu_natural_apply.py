"""Products and certificates straight from the caller's layout: grids around the
tiles' edges, every tile shape, vectors with values on closed faces, and calls
whose input and output share memory."""
import numpy as np
import pytest

import workloads as W
from oracle import geometry, operators

pytestmark = pytest.mark.gpu

# (nx, ny, nz): nodes around a 32-wide tile's edge, ny, nz around multiples of 8; the even grids
# coarsen once, so that their fine level takes the forced tile shape
GRIDS = [(30, 10, 8), (32, 8, 6), (34, 6, 18), (62, 14, 4), (31, 9, 7)]


def _workload(n):
    h = 0.1
    g = W.Grid(*n, h, 1.1 * h, 0.9 * h, (0.0, 0.0, 0.0))
    mid = (0.5 * n[0] * g.dx, 0.5 * n[1] * g.dy, 0.5 * n[2] * g.dz)
    # an ellipsoid larger than the grid along x and y: cut cells along z, open walls' neighbours elsewhere
    return W.Workload("w", g, W.ellipsoid_phi(g, mid, (0.7 * n[0] * h, 0.7 * n[1] * h, 0.47 * n[2] * h)), 3.0, 1, 0)


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("shape", [0, 1, 2, 3, 4, 5])
def test_apply_and_certify(n, shape, dm, ctx):
    import torch
    w = _workload(n)
    geom = dm.Geometry.from_workload(ctx, w)
    op = dm.Operator(ctx, geom, w.sigma, force_shape=shape, dense_coarse=0)
    assert op.stencil_shape(0) == (shape if op.num_levels > 1 else 0)
    ops = operators.DMOperators(w.grid, geometry.fractions(w.phi))
    rng = np.random.default_rng(5)
    x = rng.standard_normal(ops.a.size)                   # values on closed faces: an apply drops them
    ref = ops.apply_K(x * ops.open, w.sigma)
    tol = 1e-12 * np.max(np.abs(ref))                     # the oracle comparison of the padded applies
    got = op.apply(x)
    assert np.max(np.abs(got - ref)) < tol and np.all(got[~ops.open] == 0)
    xd = torch.from_numpy(x).cuda()
    assert np.array_equal(op.apply(xd).cpu().numpy(), got)
    assert np.max(np.abs(op.apply_noalloc(xd).cpu().numpy() - ref)) < tol
    y = xd.clone()                                        # in place
    assert np.array_equal(op.apply_noalloc(y, out=y).cpu().numpy(), got)
    B = np.stack([x * ops.open, rng.standard_normal(ops.a.size) * ops.open])
    k2 = [4.0, 9.0]
    rho, delta, rq = dm.certify(ctx, geom, k2, B)
    for i, b in enumerate(B):
        ab, kb = ops.a * b, ops.apply_K(b, 0.0)
        assert abs(rq[i] / ((b @ kb) / (b @ ab)) - 1) < 1e-12
        assert abs(rho[i] / (np.linalg.norm(kb - k2[i] * ab) / (k2[i] * np.linalg.norm(ab))) - 1) < 1e-12
        assert abs(delta[i] / (np.linalg.norm(ops.D @ ab) * min(ops.h) / np.linalg.norm(ab)) - 1) < 1e-12
