"""FP64 solves of right-hand sides of any magnitude.

Multiplying b by a power of two multiplies x and every residual by it and
changes nothing else: each operation of a solve is exact under it (alpha, beta
and the stop test are ratios, the operator scales its integers per element, and
the sums of squares follow the residual's exponent).  So the iteration counts
are those of the unscaled solve and x is its x times the power, bit for bit, at
magnitudes whose squares lie far outside FP32's exponents and inside FP64's.
One-kernel solves (up to 760 elements), the general path, batches, served
requests; a solve of a given number of iterations, which changes its operator
for such inputs, agrees in its first ten residuals to 1e-9 (each iteration's
operator and sums are within 1e-13).
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

POWERS = [-300, -200, -60, 100, 300]
SMALL, GENERAL = ((5, 4, 3), 5), ((13, 12, 5), 3)      # 60 and 780 elements


def _problem(dims, N):
    from paper_2606_12650_gb300 import Mesh
    M = Mesh(*dims, N, box_vertices(*dims, 0.05, seed=N))
    f = torch.from_numpy(normal_field(M.nL, 3)).cuda()
    b = torch.empty_like(f)
    M.rhs(f, b)
    return M, b


@pytest.mark.parametrize("dims,N", [SMALL, GENERAL])
@pytest.mark.parametrize("pre", [False, True], ids=["cg", "pcg"])
def test_solves(semlib, dims, N, pre):
    M, b = _problem(dims, N)
    solve = M.pcg_solve if pre else M.cg_solve
    x0, x = torch.empty_like(b), torch.empty_like(b)
    it0, res0 = solve(b, x0, 1e-10, 3000)
    assert res0 <= 1e-10
    for s in POWERS:
        it, res = solve(b * 2.0 ** s, x, 1e-10, 3000)
        assert (it, res) == (it0, res0), s
        assert torch.equal(x * 2.0 ** -s, x0), s
    M.free()


def test_batches(semlib):
    from paper_2606_12650_gb300 import Batch
    ps = [_problem(*SMALL), _problem(*GENERAL)]
    B = Batch([M for M, _ in ps])
    b = torch.cat([b for _, b in ps])
    x0, x = torch.empty_like(b), torch.empty_like(b)
    it0, res0 = B.solve(b, x0, 1e-10, 3000)
    assert (res0 <= 1e-10).all()
    for s in POWERS:
        it, res = B.solve(b * 2.0 ** s, x, 1e-10, 3000)
        assert (it == it0).all() and (res == res0).all(), s
        assert torch.equal(x * 2.0 ** -s, x0), s
    B.free()
    for M, _ in ps:
        M.free()


def test_served_requests(semlib):
    from paper_2606_12650_gb300 import Server
    dims, N = GENERAL
    verts = box_vertices(*dims, 0.05, seed=N)
    f = normal_field(13 * 12 * 5 * (N + 1) ** 3, 3)
    srv = Server(capacity=16, budget_gb=4.0, mode=0, tol=1e-10, maxit=3000)
    try:
        tickets = [srv.submit(*dims, N, verts, np.ldexp(f, s), srv.now(), assemble=True) for s in [0] + POWERS]
        for _ in range(1000):
            if srv.step()[2] == len(tickets):
                break
        out = []
        for tk in tickets:
            x = np.empty(len(f))
            out.append(srv.result(tk, x)[:3] + (x,))
    finally:
        srv.close()
    assert out[0][0] == 2 and out[0][2] <= 1e-10
    for s, r in zip(POWERS, out[1:]):
        assert r[:3] == out[0][:3], s
        np.testing.assert_array_equal(np.ldexp(r[3], -s), out[0][3])


@pytest.mark.parametrize("dims,N", [SMALL, GENERAL])
def test_given_number_of_iterations(semlib, dims, N):
    M, b = _problem(dims, N)
    x = torch.empty_like(b)
    h0, h = (torch.empty(11, dtype=torch.float64, device="cuda") for _ in range(2))
    M.cg_solve(b, x, 0.0, 10, h0)
    for s in POWERS:
        assert M.cg_solve(b * 2.0 ** s, x, 0.0, 10, h)[0] == 10
        np.testing.assert_allclose(np.ldexp(h.cpu().numpy(), -s), h0.cpu().numpy(), rtol=1e-9)
    M.free()


def test_iterations_past_convergence(semlib):
    """The residual of an 18-element box falls below 1e-40 of b's long before iteration 200."""
    M, b = _problem((3, 3, 2), 3)
    x0, x = torch.empty_like(b), torch.empty_like(b)
    h = torch.empty(201, dtype=torch.float64, device="cuda")
    M.cg_solve(b, x0, 1e-14, 1000)
    assert M.cg_solve(b, x, 0.0, 200, h)[0] == 200
    assert torch.isfinite(h).all() and h[200] < 1e-40 * h[0]
    assert (x - x0).abs().max() <= 1e-12 * x0.abs().max()
    M.free()
