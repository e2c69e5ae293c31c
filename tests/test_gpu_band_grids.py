"""The band smoother on unequal grids, unequal spacings and a thin slab, with bricks on both
sides of the sizes that the node kernels take: FP64 against the oracle, the lower precisions
against FP64."""
import numpy as np
import pytest

import workloads as W
from oracle import multigrid as MG

pytestmark = pytest.mark.gpu

# even, so that each coarsens; nodes of the last bricks cut along every axis; the slab has no
# node away from its walls' bands along z
GRIDS = {"ragged": ((14, 10, 22), (0.1, 0.12, 0.09)), "slab": ((34, 26, 6), (0.1, 0.09, 0.11)),
         "long": ((8, 58, 12), (0.11, 0.1, 0.1))}


def _workload(name):
    n, h = GRIDS[name]
    g = W.Grid(*n, *h, (0.0, 0.0, 0.0))
    mid = [0.49 * a * b for a, b in zip(n, h)]
    return W.Workload(name, g, W.ellipsoid_phi(g, mid, [0.46 * a * b for a, b in zip(n, h)]), 3.0, 1, 0)


@pytest.mark.parametrize("grid", sorted(GRIDS))
@pytest.mark.parametrize("brick", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_smoothing(grid, brick, dm, ctx):
    import torch
    w = _workload(grid)
    geom = dm.Geometry.from_workload(ctx, w)
    # jacobi_sweeps 1, 9 band sweeps: the oracle's step, with enough sweeps to cross a subdomain
    kw = dict(band_brick=brick, band_sweeps=9, band_sweeps_coarse=9, jacobi_sweeps=1, dense_coarse=0, autotune=0)
    op = dm.Operator(ctx, geom, w.sigma, **kw)
    levels = MG.build_vector_hierarchy(w.grid, w.phi, w.sigma, dense_coarse=0)
    assert op.num_levels == len(levels) >= 2 and levels[0].band.any()
    rng = np.random.default_rng(brick)
    for l in range(len(levels) - 1):
        lev = levels[l]
        f = rng.standard_normal(lev.mask.size) * lev.mask
        x = rng.standard_normal(lev.mask.size) * lev.mask
        ref = MG.smooth(lev, f, x, op.omega(l), 9, brick=brick)
        got = op.smooth(f, x, level=l)
        assert np.max(np.abs(got - ref)) < 1e-12 * np.max(np.abs(ref)), l   # as the smoother's parity on equal grids
    # lower precisions on the fine level: inputs exact in each of them, a sweep adds about 16
    # roundings and damps the energy norm; BF16 rounds the two stored iterates
    q = lambda v: torch.from_numpy(v).to(torch.bfloat16).double().numpy()
    mask = levels[0].mask
    x, f = q(rng.standard_normal(mask.size) * mask), q(rng.standard_normal(mask.size) * mask / min(geom.spacing)**2)
    ref = op.smooth(f, x)
    for prec, bound in (("f32", 10 * 16 * 2.0**-24), ("bf16", 2 * 4 * 2.0**-9)):
        low = dm.Operator(ctx, geom, w.sigma, precision=prec, **kw)
        low.set_omega(0, op.omega(0))
        got = low.smooth(f, x)
        assert np.linalg.norm(got - ref) < bound * np.linalg.norm(ref), prec
        assert np.all(got[mask == 0] == 0)
