"""The coarsest scalar level at its largest: a level of up to 6,000 open faces can have
up to twice as many active cells when they lie in many small components."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (ny, nz): chains of nx cells along x, one per (j, k), closed to each other.  2 x 55 x 55 =
# 6,050 and 2 x 57 x 55 = 6,270 cells lie about 6,144, three rows a thread of the inverse's
# panels and 48 KB of FP64; 2 x 77 x 77 = 11,858 is next to the largest possible
CASES = [(2, 55, 55), (2, 57, 55), (5, 37, 39), (2, 77, 77)]


@pytest.mark.parametrize("nx,ny,nz", CASES)
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
def test_cells_in_small_components(nx, ny, nz, precision, dm, ctx):
    # axes permuted so that a chain's cells lie ny * nx apart in the level's list
    gx, gy, gz = ny, nz, nx + 1 - nx % 2          # odd sides: one level
    h = 0.5
    A = [np.zeros((gz, gy, gx + 1)), np.zeros((gz, gy + 1, gx)), np.zeros((gz + 1, gy, gx))]
    A[2][1:nx] = 1.0                              # the faces within the chains
    L = np.zeros(gx * (gy + 1) * (gz + 1) + (gx + 1) * gy * (gz + 1) + (gx + 1) * (gy + 1) * gz)
    geom = dm.Geometry.from_fractions(ctx, gx, gy, gz, h, h, h, L, np.concatenate([a.ravel() for a in A]),
                                      np.ones(gx * gy * gz))
    op = dm.Operator(ctx, geom, 0.5, precision=precision, dense_coarse=6000, autotune=0)
    assert op.num_levels == 1
    # the scalar cycle is the inverse of D A D^T with the first cell of every chain pinned to zero
    S = (2 * np.eye(nx) - np.eye(nx, k=1) - np.eye(nx, k=-1)) / h**2
    S[0, 0] = S[-1, -1] = 1 / h**2
    inv = np.zeros((nx, nx))
    inv[1:, 1:] = np.linalg.inv(S[1:, 1:])
    rng = np.random.default_rng(7)
    f = np.zeros((gz, gy, gx))
    f[:nx] = rng.integers(-8, 9, (nx, gy, gx))    # exact in every storage type
    want = np.einsum("ab,bjk->ajk", inv, f[:nx])
    e = op.scalar_vcycle(f.ravel()).reshape(f.shape)
    # entries of the inverse and of the result rounded to the working precision, sums of at most four terms, and an
    # inverse by elimination in FP64
    eps = {"f64": 2.0**-53, "f32": 2.0**-24, "bf16": 2.0**-9}[precision]
    bound = lambda M, Minv, y: 16 * (eps + 2.0**-53 * np.linalg.cond(M)) * np.einsum("ab,bjk->ajk", np.abs(Minv), np.abs(y)).max()
    assert np.max(np.abs(e[:nx] - want)) <= bound(S[1:, 1:], inv, f[:nx])
    assert np.all(e[nx:] == 0)
    # the vector level of the same operator: chains of faces, A D^T D A - sigma A
    K = (2 * np.eye(nx - 1) - np.eye(nx - 1, k=1) - np.eye(nx - 1, k=-1)) / h**2 - 0.5 * np.eye(nx - 1)
    g = np.zeros((gz + 1, gy, gx))
    g[1:nx] = rng.integers(-8, 9, (nx - 1, gy, gx))
    v = op.vcycle(np.concatenate([A[0].ravel(), A[1].ravel(), g.ravel()]))[-g.size:].reshape(g.shape)
    kinv = np.linalg.inv(K)
    want = np.einsum("ab,bjk->ajk", kinv, g[1:nx])
    assert np.max(np.abs(v[1:nx] - want)) <= bound(K, kinv, g[1:nx])
