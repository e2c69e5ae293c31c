"""The coarsest level's dense inverse and product, through an operator of one level
whose V-cycle is that solve alone: sizes below, at and past the panel and tile edges."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(2, 2, 2), (3, 2, 4), (5, 4, 3), (7, 7, 7), (9, 8, 10), (11, 10, 9), (13, 12, 11)])
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
def test_one_level_vcycle_inverts_the_operator(n, precision, dm, ctx):
    w = W.box_workload(*n, lx=1.0, ly=0.9, lz=0.8, sigma=3.0)
    geom = dm.Geometry.from_workload(ctx, w)
    op = dm.Operator(ctx, geom, w.sigma, precision=precision, max_coarse=64, dense_coarse=6000)
    assert op.num_levels == 1
    _, A, _ = geom.fractions(0)
    x = np.random.default_rng(3).standard_normal(A.size) * (A > 0)
    if not x.any():
        pytest.skip("no open face")
    f = op.apply(x)
    e = op.vcycle(f)
    # K is symmetric and its condition at most about 12 n^2 / (lambda_min - sigma) < 12 * 13^2 / 3 * 10;
    # the inverse and the right-hand side are rounded to the storage precision
    eps = {"f64": 2.0**-53, "f32": 2.0**-24, "bf16": 2.0**-9}[precision]
    cond = np.linalg.norm(f) / np.linalg.norm(x) * 4.0   # ||K x|| / ||x|| bounds how far rounding f moves x, lambda_min > 1/4
    bound = 20 * eps * max(cond, 1.0) * (50 if precision == "f64" else 1)
    assert np.linalg.norm(e - x) <= bound * np.linalg.norm(x)
