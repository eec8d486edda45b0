"""The fixed-point operator's rounding errors have no sign in common.

y(x) + y(-x) is twice the part of the error that does not change sign with x.
An error of one sign everywhere comes back from a solve as A^-1 of it: with
halves upwards in the operator's last cut the solutions of 100 PCG iterations at
N = 3 were 2e-14 to 2e-13 off, ten times what errors at random leave.  Now every
cut goes away from zero at halves or meets one rarely (full significands: once
in 2^32; off-diagonal factors of a few bits: once in 2^24), so over the nodes
that part's mean is below 60 cuts x 2^-24 x 2^-45 of the mean |y|: 1e-18 with a
hundredfold allowance.  It was 4e-18 (N = 8) to 5e-16.
"""
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F64, LINES_FX = 0, 5


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_mean_error_over_nodes(semlib, N):
    from paper_2606_12650_gb300 import Mesh
    M = Mesh(13, 12, 5, N, box_vertices(13, 12, 5, 0.05, seed=N))
    u = torch.from_numpy(normal_field(M.nL, 7 + N)).cuda()
    y, z = torch.empty_like(u), torch.empty_like(u)
    M.ax(u, y)
    M.ax(-u, z)
    assert abs(float((y + z).sum())) / 2 <= 1e-18 * float(y.abs().sum())
    M.free()


def test_pcg_solution_error(semlib, oracle_mod):
    """x of 100 PCG iterations at N = 3, 900 elements, against the DFMA kernel's
    (whose rounding errors are at random): the two differ by their rounding, a
    few 1e-15; the one-signed error gave 1.7e-14."""
    from paper_2606_12650_gb300 import Mesh
    N, dims = 3, (10, 10, 9)
    M = Mesh(*dims, N, box_vertices(*dims, 0.05, seed=N))
    f = torch.from_numpy(normal_field(M.nL, 5)).cuda()
    b, xs = torch.empty_like(f), []
    M.rhs(f, b)
    old = semlib.autotune_get(F64, N)
    try:
        for choice in ((LINES_FX, 8), (1, 8)):
            semlib.autotune_set(F64, N, *choice)
            x = torch.empty_like(b)
            M.pcg_solve(b, x, 0.0, 100)
            xs.append(x)
    finally:
        semlib.autotune_set(F64, N, *old[:2])
    assert (xs[0] - xs[1]).norm() <= 6e-15 * xs[1].norm()
    M.free()
