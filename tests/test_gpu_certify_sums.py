"""Rounding of the certificates' sums: over many vectors rho, delta and the Rayleigh quotient are
within half a unit in the last place (root mean square) of their values in long double."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
Q = np.longdouble


def _split(v, dims):
    return [a.reshape(d).astype(Q) for a, d in zip(np.split(v, np.cumsum([int(np.prod(d)) for d in dims])[:-1]), dims)]


def test_errors_in_the_mean(dm, ctx):
    errors = {"rho": [], "delta": [], "rq": []}
    h = 2.0 ** -6                                  # its reciprocal is exact
    for n, seed in (((40, 36, 44), 1), ((24, 24, 24), 2), ((72, 40, 32), 3)):
        g = W.Grid(*n, h, h, h, (0.0, 0.0, 0.0))
        w = W.Workload("w", g, W.ellipsoid_phi(g, [0.49 * a * h for a in n], [0.46 * a * h for a in n]), 3.0, 1, 0)
        geom = dm.Geometry.from_workload(ctx, w)
        L, A, V = geom.fractions(0)
        nx, ny, nz = n
        fdims = [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)]
        Lx, Ly, Lz = _split(L, [(nz + 1, ny + 1, nx), (nz + 1, ny, nx + 1), (nz, ny + 1, nx + 1)])
        Ax, Ay, Az = a3 = _split(A, fdims)
        V = V.reshape(nz, ny, nx).astype(Q)
        iv, r = np.where(V > 0, 1 / np.where(V > 0, V, 1), 0), 1 / Q(h)
        low = lambda a, ax: np.diff(np.pad(a, [(1, 1) if i == ax else (0, 0) for i in range(3)]), axis=ax) * r
        high = lambda a, ax: np.diff(a, axis=ax) * r
        dot = lambda u, v: sum((x * y).sum() for x, y in zip(u, v))
        rng = np.random.default_rng(seed)
        B = rng.standard_normal((24, A.size)) * (A > 0)
        k2 = list(2000.0 + 100 * rng.random(24))
        got = dm.certify(ctx, geom, k2, B)
        for i in range(24):
            bx, by, bz = b = _split(B[i], fdims)
            ex, ey, ez = Lx * (low(bz, 1) - low(by, 0)), Ly * (low(bx, 0) - low(bz, 2)), Lz * (low(by, 2) - low(bx, 1))
            div = high(Ax * bx, 2) + high(Ay * by, 1) + high(Az * bz, 0)
            psi = iv * div
            kb = [high(ez, 1) - high(ey, 0) - Ax * low(psi, 2), high(ex, 0) - high(ez, 2) - Ay * low(psi, 1),
                  high(ey, 2) - high(ex, 1) - Az * low(psi, 0)]
            kb = [np.where(a > 0, k, 0) for a, k in zip(a3, kb)]
            ab = [a * x for a, x in zip(a3, b)]
            norm, kk = np.sqrt(dot(ab, ab)), Q(k2[i])
            res = [x - kk * y for x, y in zip(kb, ab)]
            want = {"rho": np.sqrt(dot(res, res)) / (kk * norm), "delta": np.sqrt((div * div).sum()) * Q(h) / norm,
                    "rq": dot(b, kb) / dot(b, ab)}
            for k, v in zip(("rho", "delta", "rq"), got):
                errors[k].append(float((Q(v[i]) - want[k]) / want[k]))
    # two or three roundings of at most half a unit each, spread evenly, and sums that add little to them
    for k, e in errors.items():
        assert np.sqrt(np.mean(np.square(e))) <= 2.0 ** -53, k
