"""CG solves of a given number of iterations (tol = 0) keep their iterates.

After CG has converged on the operator's largest eigenvector, rounding brings
that component back, enlarged by up to 1e7 by iteration 100: the iterate is
then a property of the arithmetic.  The stored solutions and histories of two
such boxes (3 x 3 x 2 elements, vertices moved by 5 %) were recorded from the
double-word operator with the update of every copy; the fixed-point operator
with the update by owner rows gives x 3e-9 and 1.4e-6 away.  The bound is the
1e-9 that FP64 results may move by; the same operations in the same order
differ by nothing.
"""
import os

import numpy as np
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "cg_steps_3x3x2.npz")


@pytest.mark.parametrize("N,seed", [(6, 5), (9, 1)])
def test_iterates_after_100_iterations(semlib, N, seed):
    from paper_2606_12650_gb300 import Mesh
    ref = np.load(GOLDEN)
    M = Mesh(3, 3, 2, N, box_vertices(3, 3, 2, 0.05, seed=seed))
    f = torch.from_numpy(normal_field(M.nL, 100 + seed)).cuda()
    b = torch.empty_like(f)
    M.rhs(f, b)
    for _ in range(2):                     # a first solve, and one from its captured graph
        x = torch.full_like(b, float("nan"))
        h = torch.full((101,), float("nan"), dtype=torch.float64, device="cuda")
        it, _ = M.cg_solve(b, x, 0.0, 100, h)
        assert it == 100
        for got, want in ((x, ref[f"x_{N}_{seed}"]), (h, ref[f"h_{N}_{seed}"])):
            assert np.linalg.norm(got.cpu().numpy() - want) <= 1e-9 * np.linalg.norm(want)
    M.free()
