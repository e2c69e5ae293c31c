"""One network trained on several geometries in turn: a step's loss and gradient are those of a
network that has seen nothing else (its kept work vectors hold nothing of another geometry)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _problem(dm, ctx, n, fill, seed):
    g = W.Grid(*n, 0.1, 0.1, 0.1, (0.0, 0.0, 0.0))
    mid = [0.05 * v for v in n]
    w = W.Workload("w", g, W.ellipsoid_phi(g, mid, [fill * v for v in mid]), 2.0, 1, 0)
    geom = dm.Geometry.from_workload(ctx, w)
    op = dm.Operator(ctx, geom, 2.0, precision="f32", dense_coarse=6000, autotune=0)
    A = geom.fractions(0)[1]
    return op, np.random.default_rng(seed).standard_normal(A.size) * (A > 0)


def test_geometries_in_turn(dm, ctx):
    # the same grid filled more and less, and its sides exchanged (the same number of nodes)
    problems = [_problem(dm, ctx, n, fill, 3 + i) for i, (n, fill) in
                enumerate([((72, 12, 24), 0.95), ((72, 12, 24), 0.4), ((24, 12, 72), 0.9), ((72, 24, 12), 0.5)])]
    net = dm.Learned(ctx, seed=5)
    w0 = net.get_weights()
    for op, r in problems * 2:
        fresh = dm.Learned(ctx, seed=5)
        fresh.set_weights(w0)
        net.set_weights(w0)
        want, got = fresh.train_step(op, r), net.train_step(op, r)
        # (NaN where a nearly empty cut cell takes FP32's range, for both alike)
        assert np.array_equal(got[0], want[0], equal_nan=True) and np.array_equal(got[1], want[1], equal_nan=True)
        fresh.close()
    net.close()
