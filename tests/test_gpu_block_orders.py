"""Inner solves whose last step of the correction is left to the next operator
launch, and solves of the batch engine that run one block per item.

Boxes one element thick have no copies in a direction, ragged ones leave warps
and blocks partly empty, and many elements per problem take the sum of <p, A p>
through one or several blocks.  A solution must pass the oracle's residual test
at its tolerance (1.5x slack for the different rounding of the two FP64
operators); with FP32 factors an inner solve to 1e-3 contracts the true residual
by about that, so 1e-9 takes three outer steps and one more at most.
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F64, F32G32, F32G16 = 0, 1, 2
COLUMNS, LINES, PERSISTENT, LINES_ST, LINES_FX = 0, 1, 2, 4, 5
TOL = 1e-9


@pytest.mark.parametrize("dims", [(1, 1, 5), (6, 1, 1), (1, 7, 2), (17, 3, 2)])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_mixed_on_thin_and_ragged_boxes(semlib, oracle_mod, dims, N):
    from paper_2606_12650_gb300 import Mesh
    verts = box_vertices(*dims, 0.05, seed=N)
    P, M = oracle_mod.Problem(*dims, N, verts), Mesh(*dims, N, verts)
    b_ref = P.mask(P.gs(normal_field(P.nL, 5 + N)))
    b = torch.from_numpy(b_ref).cuda()
    for gprec, kind in ((0, F32G32), (1, F32G16)):
        old = semlib.autotune_get(kind, N)
        try:
            for choice in ((LINES, 1), (LINES, max(1, 256 // (N + 1) ** 2)), (PERSISTENT, 0), (LINES_ST, 2)):
                semlib.autotune_set(kind, N, *choice)
                x = torch.full_like(b, float("nan"))
                inner, outer, res = M.cg_mixed(b, x, TOL, 50, 1e-3, 100000, gprec)
                if not b_ref.any():
                    assert not x.cpu().numpy().any()
                    continue
                assert res <= TOL and P.true_residual(b_ref, x.cpu().numpy()) <= 1.5 * TOL, choice
                if gprec == 0:
                    assert outer <= 4, choice
        finally:
            semlib.autotune_set(kind, N, *old[:2])
    M.free()


@pytest.mark.parametrize("dims", [(16, 16, 8), (3, 683, 1), (14, 13, 13), (84, 84, 85)])
def test_sums_over_many_blocks(semlib, dims):
    """2048 parts (one block), 2049 and 2366 (several), 599760 (several parts per thread)."""
    from paper_2606_12650_gb300 import Mesh
    N = 1 if dims != (3, 683, 1) else 2
    M = Mesh(*dims, N, box_vertices(*dims, 0.0))
    f = torch.from_numpy(normal_field(M.nL, 3)).cuda()
    b = torch.empty_like(f)
    M.rhs(f, b)
    old = semlib.autotune_get(F32G32, N)
    counts = []
    try:
        for epb in (1, 32):
            semlib.autotune_set(F32G32, N, LINES, epb)
            x = torch.empty_like(b)
            inner, outer, res = M.cg_mixed(b, x, TOL, 50, 1e-3, 100000, 0)
            assert res <= TOL and outer <= 4
            counts.append(inner)
    finally:
        semlib.autotune_set(F32G32, N, *old[:2])
    assert abs(counts[0] - counts[1]) <= 0.02 * counts[1] + 2
    M.free()


@pytest.mark.parametrize("mode,kind,choices", [(0, F64, [(LINES, 4), (LINES_FX, 4)]),
                                               (1, F32G16, [(PERSISTENT, 0), (LINES, 2)])])
@pytest.mark.parametrize("first", [0, 1])
def test_table_change_in_mid_solve(semlib, oracle_mod, mode, kind, choices, first):
    """A request in mid-solve keeps its operator when the table changes under
    it, also when a new request of its order joins."""
    from paper_2606_12650_gb300 import Server
    N, dims = 5, (4, 3, 3)
    reqs = []
    for k in range(2):
        verts = box_vertices(*dims, 0.05, seed=k)
        P = oracle_mod.Problem(*dims, N, verts)
        reqs.append((P, verts, normal_field(P.nL, 40 + k)))
    old = semlib.autotune_get(kind, N)
    srv = Server(capacity=16, budget_gb=4.0, mode=mode, tol=1e-8, K=8)
    try:
        semlib.autotune_set(kind, N, *choices[first])
        tickets = [srv.submit(*dims, N, reqs[0][1], reqs[0][2], srv.now(), assemble=True)]
        srv.step()
        semlib.autotune_set(kind, N, *choices[1 - first])
        tickets.append(srv.submit(*dims, N, reqs[1][1], reqs[1][2], srv.now(), assemble=True))
        for _ in range(10000):
            if srv.step()[2] == 2:
                break
        for tk, (P, _, f) in zip(tickets, reqs):
            x = torch.empty(P.nL, dtype=torch.float64, device="cuda")
            assert srv.result(tk, x)[0] == 2
            b = P.mask(P.gs(f))
            assert P.true_residual(b, x.cpu().numpy()) <= 1.5e-8
    finally:
        semlib.autotune_set(kind, N, *old[:2])
        srv.close()
