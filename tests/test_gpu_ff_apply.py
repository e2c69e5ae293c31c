"""The float-float apply and the compact preconditioned vectors: grids around the
tiles' edges, unequal and equal spacings, magnetic walls, every storage type."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import geometry, operators

pytestmark = pytest.mark.gpu


def _w(n, h, walls=("pec",) * 6):
    g = W.Grid(*n, *h, (0.0, 0.0, 0.0))
    mid = [0.48 * a * b for a, b in zip(n, h)]
    # wide along x, so that whole 32-node rows lie inside the vacuum
    w = W.Workload("w", g, W.ellipsoid_phi(g, mid, (1.2 * n[0] * h[0], 0.46 * n[1] * h[1], 0.45 * n[2] * h[2])), 2.0, 1, 0)
    return dataclasses.replace(w, walls=walls)


CASES = {
    "cube70": lambda: _w((70, 18, 16), (0.1, 0.1, 0.1)),
    "flat98": lambda: _w((98, 10, 20), (0.1, 0.11, 0.07)),
    "pmc64": lambda: _w((64, 16, 18), (0.1, 0.1, 0.1), ("pmc", "pec", "pmc", "pec", "pec", "pec")),
    "tiny": lambda: _w((3, 4, 2), (0.2, 0.2, 0.3)),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
def test_apply_ff_and_solve(name, precision, dm, ctx):
    w = CASES[name]()
    geom = dm.Geometry.from_workload(ctx, w)
    op = dm.Operator(ctx, geom, 0.3, precision=precision, dense_coarse=6000)
    ops = operators.DMOperators(w.grid, geometry.fractions(w.phi, walls=w.walls))
    rng = np.random.default_rng(2)
    x = rng.standard_normal(ops.a.size) * ops.open
    ref = ops.apply_K(x, 0.3)
    # as the float-float apply's comparison with the oracle: about 48 bits an operation
    assert np.max(np.abs(op.apply_ff(x) - ref)) < 1e-12 * np.max(np.abs(ref))
    # the iterations apply the operator to the V-cycle's own type and form the solution from it
    sol, it, rr = op.solve(ref, tol=1e-10)
    assert rr <= 1e-9
    r = np.linalg.norm(ops.apply_K(sol, 0.3) - ref) / np.linalg.norm(ref)
    assert abs(r - rr) < 1e-12 and np.all(sol[~ops.open] == 0)
