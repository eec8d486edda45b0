"""<p, A p> of the fixed-point operator for vectors that make its sums largest.

One CG iteration from b gives x = alpha b with alpha = <b, b> / <b, A b>: nodes of
alternating and of random sign and all of one sign, in the one-kernel solve
and (780 elements) the general one, against the oracle's operator.  The
operator is within 1e-13 of the oracle's per element and the sums are exact or
FP64, so alpha is within 1e-12.
"""
import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 2, 2), (13, 12, 5)])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_first_step(semlib, oracle_mod, dims, N):
    from paper_2606_12650_gb300 import Mesh
    nx, ny, nz, n = *dims, N + 1
    verts = box_vertices(*dims, 0.05, seed=N)
    P, M = oracle_mod.Problem(*dims, N, verts), Mesh(*dims, N, verts)
    I, J, K = (np.arange(m)[:, None] * N + np.arange(n)[None, :] for m in dims)
    shape = (nz, ny, nx, n, n, n)
    at = lambda v, a, b: np.broadcast_to(v.reshape([v.shape[0] if q == a else v.shape[1] if q == b else 1 for q in range(6)]), shape)
    i, j, k = at(I, 2, 5), at(J, 1, 4), at(K, 0, 3)
    lattice = np.sign(np.random.default_rng(N).standard_normal((nz * N + 1, ny * N + 1, nx * N + 1)))
    for field in ((-1.0) ** (i + j + k), lattice[k, j, i], np.ones(shape)):
        b = P.mask(np.ascontiguousarray(field.reshape(-1)))
        if not b.any():
            continue
        Ab = P.ax_local(b)
        x = torch.empty(P.nL, dtype=torch.float64, device="cuda")
        M.cg_solve(torch.from_numpy(b).cuda(), x, 1e-300, 1)
        alpha = (P.c * b * b).sum() / (b * Ab).sum()
        np.testing.assert_allclose(x.cpu().numpy(), alpha * b, rtol=1e-12, atol=0)
    M.free()
