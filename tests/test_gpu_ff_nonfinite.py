"""The float-float apply of a vector with a non-finite entry: covered edges and cells pass it
on to no face, so it reaches only the faces that share an uncovered edge or cell with its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _reach(n, L, V):
    """For every face the faces that share an edge with L > 0 or a cell with V > 0 with it."""
    nx, ny, nz = n
    fdims = [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)]
    edims = [(nz + 1, ny + 1, nx), (nz + 1, ny, nx + 1), (nz, ny + 1, nx + 1)]
    size = lambda dims: np.concatenate([[0], np.cumsum([int(np.prod(d)) for d in dims])])
    foff, eoff = size(fdims), size(edims)
    face = [foff[c] + np.arange(foff[c + 1] - foff[c]).reshape(d) for c, d in enumerate(fdims)]
    groups = []
    for c, d in enumerate(edims):
        for q, node in enumerate(np.ndindex(*d)):             # (k, j, i)
            if not L[eoff[c] + q] > 0:
                continue
            group = []
            for a in ((c + 1) % 3, (c + 2) % 3):              # faces normal to a, on both sides across the third axis
                for s in (0, 1):
                    m = list(node)
                    m[2 - (3 - c - a)] -= s
                    if all(0 <= v < w for v, w in zip(m, face[a].shape)):
                        group.append(face[a][tuple(m)])
            groups.append(group)
    for q, (k, j, i) in enumerate(np.ndindex(nz, ny, nx)):
        if V[q] > 0:
            groups.append([face[0][k, j, i], face[0][k, j, i + 1], face[1][k, j, i], face[1][k, j + 1, i],
                           face[2][k, j, i], face[2][k + 1, j, i]])
    reach = {}
    for g in groups:
        for a in g:
            reach.setdefault(a, set()).update(g)
    return face, reach


@pytest.mark.parametrize("n,h", [((9, 7, 11), (0.1, 0.1, 0.1)), ((35, 9, 5), (0.1, 0.11, 0.09))])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_entries_stay_within_reach(n, h, bad, dm, ctx):
    rng = np.random.default_rng(4)
    nx, ny, nz = n
    E = nx * (ny + 1) * (nz + 1) + (nx + 1) * ny * (nz + 1) + (nx + 1) * (ny + 1) * nz
    L = rng.choice([0.0, 0.0, 0.5, 1.0], E)
    V = rng.choice([0.0, 0.5, 1.0], nx * ny * nz)
    face, reach = _reach(n, L, V)
    A = rng.choice([0.0, 0.5, 1.0, 1.0], face[2].ravel()[-1] + 1)
    for c, f in enumerate(face):                              # closed walls
        f = np.moveaxis(f, 2 - c, 0)
        A[f[0].ravel()] = A[f[-1].ravel()] = 0.0
    geom = dm.Geometry.from_fractions(ctx, *n, *h, L, A, V)
    op = dm.Operator(ctx, geom, -3.0, dense_coarse=6000, autotune=0)
    x = rng.standard_normal(A.size) * (A > 0)
    clean = op.apply_ff(x)
    for q in rng.permutation(np.flatnonzero(A > 0))[:32]:
        xb = x.copy()
        xb[q] = bad
        far = np.ones(A.size, bool)
        far[list(reach.get(q, set()) | {q})] = False
        y = op.apply_ff(xb)
        assert np.array_equal(y[far], clean[far])
