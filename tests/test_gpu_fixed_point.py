"""The fixed-point FP64 operator where its integer scales could go wrong.

Per element its values are 64-bit integers on one power-of-two scale, so the
inputs that matter are the largest sums (signs aligned with a row of D),
elements of very different magnitude side by side, zero elements and elements
that hold a NaN or an infinity.  Each element is compared with the oracle's
on its own: within 1e-13 of its max |y|, the bar of the FP64 operator (the
dropped parts are ~20 units of 2^-61 of the largest possible |y|, and max |y|
is above 2^-14 of that for these inputs: < 2e-14).
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F64, LINES_FX = 0, 5


def _err_per_element(y, ref, E):
    y, ref = y.reshape(E, -1), ref.reshape(E, -1)
    return np.abs(y - ref).max(axis=1) / np.abs(ref).max(axis=1)


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_extreme_inputs(semlib, oracle_mod, N):
    from paper_2606_12650_gb300 import Mesh
    nx, ny, nz, n = 3, 5, 7, N + 1
    E = nx * ny * nz
    verts = box_vertices(nx, ny, nz, 0.05, seed=N)
    P, M = oracle_mod.Problem(nx, ny, nz, N, verts), Mesh(nx, ny, nz, N, verts)
    old = semlib.autotune_get(F64, N)
    rng = np.random.default_rng(N)
    signs = np.sign(P.D)                                  # row i: the input that makes (D u)_i largest
    aligned = np.empty((E, n, n, n))
    for e in range(E):
        r, s, t = (signs[rng.integers(n)] for _ in range(3))
        aligned[e] = t[:, None, None] * s[None, :, None] * r[None, None, :]
    random = normal_field(P.nL, 7 + N).reshape(E, -1)
    scaled = np.ldexp(random, rng.integers(-200, 200, size=(E, 1)))
    try:
        for epb in (1, 3, max(1, 256 // n ** 2)):
            semlib.autotune_set(F64, N, LINES_FX, epb)
            for x in (aligned, np.sign(random), scaled):
                x = np.ascontiguousarray(x.reshape(-1))
                yd = torch.full((P.nL,), float("nan"), dtype=torch.float64, device="cuda")
                M.ax(torch.from_numpy(x).cuda(), yd)
                err = _err_per_element(yd.cpu().numpy(), P.ax_local(x), E)
                assert (err < 1e-13).all(), epb
            x = random.copy()
            x[4] = 0.0
            x[9, 3] = np.nan
            x[11, 2] = np.inf
            x = x.reshape(-1)
            yd = torch.full((P.nL,), 7.0, dtype=torch.float64, device="cuda")
            M.ax(torch.from_numpy(x).cuda(), yd)
            y = yd.cpu().numpy().reshape(E, -1)
            assert np.array_equal(y[4], np.zeros(n ** 3))
            assert np.isnan(y[9]).all() and np.isnan(y[11]).all()
            rest = [e for e in range(E) if e not in (4, 9, 11)]
            ref = P.ax_local(random.reshape(-1)).reshape(E, -1)[rest]
            assert (np.abs(y[rest] - ref).max(axis=1) < 1e-13 * np.abs(ref).max(axis=1)).all()
    finally:
        semlib.autotune_set(F64, N, old[0], old[1])
        M.free()
