"""The coarsest solve of the lower precisions on a right-hand side they hold exactly: within the
rounding of the result, far below the result itself."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(2, 2, 2), (5, 4, 3), (7, 7, 7), (9, 8, 10), (13, 12, 11)])
@pytest.mark.parametrize("precision", ["f32", "bf16"])
def test_one_level_vcycle_against_fp64(n, precision, dm, ctx):
    import torch
    w = W.box_workload(*n, lx=1.0, ly=0.9, lz=0.8, sigma=3.0)
    geom = dm.Geometry.from_workload(ctx, w)
    ops = {p: dm.Operator(ctx, geom, w.sigma, precision=p, max_coarse=64, dense_coarse=6000) for p in ("f64", precision)}
    assert all(o.num_levels == 1 for o in ops.values())
    A = geom.fractions(0)[1]
    f = torch.from_numpy(np.random.default_rng(3).standard_normal(A.size) * (A > 0)).to(torch.bfloat16).double().numpy()
    if not f.any():
        pytest.skip("no open face")
    want, got = ops["f64"].vcycle(f), ops[precision].vcycle(f)   # (FP64: held to the operator by its own test)
    # the result rounded to the storage type; the inverse to FP32, ||M^-1|| <= 1 / (lambda_min - sigma) with the
    # box's lambda_min - sigma > 1 by its size, so at most sqrt(3) 2^-24 ||f|| and a little for FP64
    eps = {"f32": 2.0**-24, "bf16": 2.0**-9}[precision]
    bound = eps * np.linalg.norm(want) + 2 * 2.0**-24 * np.sqrt(f.size) * np.linalg.norm(f)
    assert bound < 0.05 * np.linalg.norm(want)
    assert np.linalg.norm(got - want) <= bound
