"""Whole CG and PCG solves in one kernel (problems of up to five elements per
SM) against the general path, which every other operator variant takes.

Block counts around the exchange's limits (32 blocks and their neighbours, whole
and partial groups) and the rule's own limit (760 elements on 152 SMs), boxes
one element thick, every order.  Both paths run the same recurrences, so their
histories differ by rounding alone: the first entries, before rounding grows
with the iterations, agree to 1e-9 relative (each iteration's operator and sums
are within 1e-13, and amplification over ten iterations is far below 1e4), the
iteration counts at 1e-8 by two at most, and the solution passes the oracle's
residual test with 1.5x slack.
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F64, LINES = 0, 1


def _both(semlib, M, b, N, solve, tol, maxit):
    old = semlib.autotune_get(F64, N)
    out = []
    try:
        for choice in (old[:2], (LINES, max(1, 256 // (N + 1) ** 2))):
            semlib.autotune_set(F64, N, *choice)
            x = torch.full_like(b, float("nan"))
            h = torch.full((maxit + 1,), float("nan"), dtype=torch.float64, device="cuda")
            it, res = solve(M)(b, x, tol, maxit, h)
            out.append((it, res, x.cpu().numpy(), h.cpu().numpy()))
    finally:
        semlib.autotune_set(F64, N, *old[:2])
    return out


@pytest.mark.parametrize("pre", [False, True], ids=["cg", "pcg"])
@pytest.mark.parametrize("dims,N", [((1, 1, 5), 2), ((7, 1, 2), 3), ((4, 4, 2), 7), ((11, 3, 1), 5), ((4, 4, 4), 9),
                                    ((13, 5, 1), 8), ((3, 11, 3), 6), ((4, 8, 4), 4), ((19, 6, 4), 3),
                                    ((19, 6, 4), 1), ((5, 4, 3), 1), ((19, 8, 5), 3),
                                    ((19, 2, 8), 9), ((19, 2, 16), 7), ((20, 19, 2), 2)])
def test_matches_the_general_path(semlib, oracle_mod, dims, N, pre):
    from paper_2606_12650_gb300 import Mesh
    verts = box_vertices(*dims, 0.05, seed=N)
    P, M = oracle_mod.Problem(*dims, N, verts), Mesh(*dims, N, verts)
    b_ref = P.mask(P.gs(normal_field(P.nL, 3 + N)))
    b = torch.from_numpy(b_ref).cuda()
    solve = (lambda m: m.pcg_solve) if pre else (lambda m: m.cg_solve)
    (it, res, x, h), (it2, _, _, h2) = _both(semlib, M, b, N, solve, 1e-8, 5000)
    if not b_ref.any():
        assert it == 0 and not x.any()
        return
    k = min(it, it2, 10) + 1
    np.testing.assert_allclose(h[:k], h2[:k], rtol=1e-9, atol=1e-9 * h[0])
    assert abs(it - it2) <= 2 and res <= 1e-8 and np.isfinite(h[:it + 1]).all() and np.isnan(h[it + 1:]).all()
    assert P.true_residual(b_ref, x) <= 1.5e-8
    M.free()


@pytest.mark.parametrize("maxit", [0, 1, 2, 7])
def test_iteration_limits(semlib, oracle_mod, maxit):
    """An odd and an even last iteration (w alternates between two buffers), no
    iteration at all, and a solve after each on the same problem."""
    from paper_2606_12650_gb300 import Mesh
    dims, N = (3, 4, 3), 5
    verts = box_vertices(*dims, 0.05, seed=N)
    P, M = oracle_mod.Problem(*dims, N, verts), Mesh(*dims, N, verts)
    b_ref = P.mask(P.gs(normal_field(P.nL, 3)))
    b = torch.from_numpy(b_ref).cuda()
    (it, _, x, h), (it2, _, x2, h2) = _both(semlib, M, b, N, lambda m: m.cg_solve, 0.0, maxit)
    assert it == it2 == maxit
    np.testing.assert_allclose(h, h2, rtol=1e-9)
    np.testing.assert_allclose(x, x2, rtol=0, atol=1e-9 * max(1e-300, np.abs(x2).max()))
    x = torch.empty_like(b)
    M.cg_solve(b, x, 1e-8, 5000)
    assert P.true_residual(b_ref, x.cpu().numpy()) <= 1.5e-8
    M.free()


def test_more_iterations_than_one_launch(semlib, oracle_mod):
    """1024 iterations a launch: a long thin box takes several."""
    from paper_2606_12650_gb300 import Mesh
    dims, N = (1, 1, 400), 3
    verts = box_vertices(*dims, 0.05, seed=N)
    P, M = oracle_mod.Problem(*dims, N, verts), Mesh(*dims, N, verts)
    b_ref = P.mask(P.gs(normal_field(P.nL, 3)))
    b = torch.from_numpy(b_ref).cuda()
    (it, res, x, h), (it2, _, _, _) = _both(semlib, M, b, N, lambda m: m.cg_solve, 1e-4, 6000)
    assert it > 1024 and abs(it - it2) <= 0.02 * it2 and res <= 1e-4
    assert np.isfinite(h[:it + 1]).all() and P.true_residual(b_ref, x) <= 1.5e-4
    M.free()
