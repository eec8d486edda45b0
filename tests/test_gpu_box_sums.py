"""The box-structured gather-scatter with and without the mask, the update by
owner rows, and the grid sums, at sizes where their enumerations could go wrong.

Boxes one element thick have no copies in a direction, and element counts off
the multiples of a warp's group leave lanes idle.  The gather-scatter adds in
ascending local order, so it equals the oracle's sum bit for bit, and the fused
form equals the separate calls.  Grid sums change from one level to two beyond
1024 blocks; histories of two operator variants with different block counts run
the same recurrences and differ by rounding alone, so their first ten entries
agree to 1e-9 relative (each operator and sum is within 1e-13).
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F64, LINES, LINES_FX = 0, 1, 5


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 1, 9), (7, 1, 1), (1, 5, 3), (2, 2, 2), (5, 4, 3)])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_gather_scatter(semlib, oracle_mod, dims, N):
    from paper_2606_12650_gb300 import Mesh
    verts = box_vertices(*dims, 0.05, seed=N)
    P, M = oracle_mod.Problem(*dims, N, verts), Mesh(*dims, N, verts)
    u_ref = normal_field(P.nL, 11 + N)
    u = torch.from_numpy(u_ref).cuda()
    v = u.clone()
    M.gs(v)
    np.testing.assert_array_equal(v.cpu().numpy(), P.gs(u_ref))
    y, z = torch.empty_like(u), torch.empty_like(u)
    M.ax(u, y)
    M.gs(y)
    M.mask(y)
    M.axg(u, z)
    assert torch.equal(y, z)
    M.free()


@pytest.mark.parametrize("pre", [False, True], ids=["cg", "pcg"])
@pytest.mark.parametrize("dims", [(31, 33, 1), (32, 32, 1), (41, 25, 1), (33, 32, 2), (13, 12, 11)])
@pytest.mark.parametrize("N", [1, 2, 4])
def test_grid_sums_and_owner_rows(semlib, dims, N, pre):
    """1023, 1024, 1025, 2112 and 1716 elements, one per block, against a few per block."""
    from paper_2606_12650_gb300 import Mesh
    M = Mesh(*dims, N, box_vertices(*dims, 0.05, seed=N))
    f = torch.from_numpy(normal_field(M.nL, 3)).cuda()
    b = torch.empty_like(f)
    M.rhs(f, b)
    old = semlib.autotune_get(F64, N)
    hists = []
    try:
        for choice in ((LINES_FX, 1), (LINES, 4)):
            semlib.autotune_set(F64, N, *choice)
            x = torch.empty_like(b)
            h = torch.empty(11, dtype=torch.float64, device="cuda")
            (M.pcg_solve if pre else M.cg_solve)(b, x, 0.0, 10, h)
            hists.append(h.cpu().numpy())
    finally:
        semlib.autotune_set(F64, N, *old[:2])
    if hists[1][0] == 0.0:      # no interior node (N = 1, one element thick)
        assert not hists[0][0]
        return
    np.testing.assert_allclose(hists[0], hists[1], rtol=1e-9, atol=1e-9 * hists[1][0])
    M.free()
