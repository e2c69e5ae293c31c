"""The band smoother's node kernels: every class of subdomain size and every
precision against the FP64 kernels, which test_gpu_operators.py holds to the oracle."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# 16^3: few subdomains, one launch (FP32) and clusters of eight (FP64); 64^3:
# classes launched side by side; a thin slab and a 13 x 11 x 9 grid: bricks cut by
# the grid's end; bricks below 8: boxes smaller than the local layout
GRIDS = {
    "sphere16": lambda: W.sphere_workload(16, offset_seed=W.SEED_BASE + 1, sigma=7.0),
    "ellipsoid64": lambda: W.ellipsoid_workload(64, seed=W.SEED_BASE + 3, sigma=5.0),
    "ragged13x11x9": lambda: W.sphere_workload(13, offset_seed=5, sigma=6.0),
}


@pytest.mark.parametrize("grid,brick", [("sphere16", 8), ("ellipsoid64", 8), ("ellipsoid64", 3), ("ragged13x11x9", 8)])
@pytest.mark.parametrize("precision", ["f32", "bf16"])
def test_low_precision_smoothing_follows_fp64(grid, brick, precision, dm, ctx):
    w = GRIDS[grid]()
    geom = dm.Geometry.from_workload(ctx, w)
    sweeps = 24
    ops = {p: dm.Operator(ctx, geom, w.sigma, precision=p, band_brick=brick, band_sweeps=sweeps, dense_coarse=0)
           for p in ("f64", precision)}
    if ops["f64"].num_levels < 2:
        pytest.skip("one level: nothing is smoothed")
    _, A, _ = geom.fractions(0)
    rng = np.random.default_rng(17)
    # inputs exact in both storage types, so that only the arithmetic differs
    import torch
    q = lambda v: torch.from_numpy(v).to(torch.bfloat16).double().numpy()
    x = q(rng.standard_normal(A.size) * (A > 0))
    h = min(geom.spacing)
    f = q(rng.standard_normal(A.size) * (A > 0) / h**2)
    ops[precision].set_omega(0, ops["f64"].omega(0))
    got, ref = ops[precision].smooth(f, x), ops["f64"].smooth(f, x)
    # x enters at size 1 and f at 1/h^2.  A damped sweep, omega / lambda_max of a
    # symmetrisable operator, does not amplify rounding in the energy norm; each of
    # the 2 + 24 sweeps adds about 16 roundings of eps.  BF16 rounds the three stored
    # iterates (eps 2^-9) instead.
    eps = 2.0**-24 if precision == "f32" else 2.0**-9
    bound = (26 * 16 if precision == "f32" else 3 * 4) * eps
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < bound, (err, bound)
    assert np.all(got[A == 0] == 0)
