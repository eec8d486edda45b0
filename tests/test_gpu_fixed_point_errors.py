"""The fixed-point operator's error on smooth inputs, wide ratios and stretched
elements, against the same factors in extended precision.

Its roundings are absolute on the element's scale.  In units of the integers a
contraction of n terms is off by n / 4 (dropped low products) + n / 32
(coefficients) + 1/2, below 4 for n <= 10; relative to the largest possible U
(2^59 and up), W (2^58.6) and Y (2^59, three directions) the three phases add
2^-57 + 2^-57.6 + 2^-55.4 < 2^-54.8, and each of the four scales (x, D, G, D^T) is a
power of two up to twice too wide: below 2^-50.8 of the largest |y| that the
element's max |x| and max |G| allow, 9 R^2 max|x| max|G| with R the largest row sum
of |D| and (for D^T) of its columns.  y itself is rounded to 51 bits of the largest on
the thread's line.  That holds for every input; relative to max|y| the error of
smooth inputs, whose y is a small remainder of those sums, is larger (and
FP64's is too).
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sides", [(1, 1, 1), (1000, 1, 1), (1000, 30, 1)])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_error_bound(semlib, oracle_mod, N, sides):
    from paper_2606_12650_gb300 import Mesh
    nx, ny, nz, n, E = 2, 2, 1, N + 1, 4
    verts = np.ascontiguousarray(box_vertices(nx, ny, nz, 0.05, seed=N) * np.array(sides, dtype=float))
    D = np.asarray(oracle_mod.Problem(nx, ny, nz, N, verts).D)
    M = Mesh(nx, ny, nz, N, verts)
    G, B, X = (torch.empty(M.nL * m, dtype=torch.float64, device="cuda") for m in (6, 1, 3))
    M.geom(G, B)
    M.nodes(X)
    g = G.cpu().numpy().reshape(E, n, n, n, 6).astype(np.longdouble)
    pos = X.cpu().numpy().reshape(-1, 3) / np.array(sides)
    r = np.random.default_rng(N)
    inputs = [np.prod(np.sin(np.pi * pos / 4), axis=1), np.prod(np.sin(np.pi * pos / 16), axis=1),
              1.0 + 1e-6 * r.standard_normal(M.nL), r.standard_normal(M.nL) * np.exp2(r.integers(-60, 1, M.nL)),
              r.standard_normal(M.nL)]
    Dl = D.astype(np.longdouble)
    along = lambda u, axis, Q: np.moveaxis(np.tensordot(u, Q, axes=(axis, 1)), -1, axis)
    R2 = np.abs(D).sum(axis=1).max() * np.abs(D).sum(axis=0).max()
    for x in inputs:
        u = x.reshape(E, n, n, n).astype(np.longdouble)
        d = [along(u, a, Dl) for a in (3, 2, 1)]
        w = [sum(g[..., q] * d[b] for b, q in enumerate(row)) for row in ((0, 1, 2), (1, 3, 4), (2, 4, 5))]
        ref = sum(along(w[a], 3 - a, Dl.T) for a in range(3)).reshape(E, -1)
        y = torch.empty(M.nL, dtype=torch.float64, device="cuda")
        M.ax(torch.from_numpy(x).cuda(), y)
        err = np.abs(y.cpu().numpy().reshape(E, -1) - ref).max(axis=1)
        most = 9 * R2 * np.abs(x).reshape(E, -1).max(axis=1) * np.abs(g).reshape(E, -1).max(axis=1)
        assert (err <= 2.0 ** -50.8 * most + 2.0 ** -52 * np.abs(ref).max(axis=1)).all()
    M.free()
