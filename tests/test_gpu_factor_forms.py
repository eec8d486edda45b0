"""Integer and double-word factors of one problem when only one form fits.

Operator calls and solves to a tolerance use the integer form, solves of a given
number of iterations the double-word form (48 bytes a node each).  With an HBM
budget that leaves room for one of them, each call makes its own again in the
other's place, and results do not change.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHILD = """
import sys
import torch
from paper_2606_12650_gb300 import Mesh, sem
from paper_2606_12650_gb300.inputs import box_vertices, normal_field
nL = 10 ** 3 * 512
if sys.argv[1] == "one":
    sem.init(["--device=0", "--hbm-budget=%.9f" % (nL * (96 + 48 + 30) / 1e9)])   # 96: G, mass, weights, vectors; 30: lists, sums
else:
    sem.init(["--device=0"])
torch.cuda.set_stream(sem.stream())
M = Mesh(10, 10, 10, 7, box_vertices(10, 10, 10, 0.05, seed=1))
f = torch.from_numpy(normal_field(M.nL, 3)).cuda()
b, y, x = torch.empty_like(f), torch.empty_like(f), torch.empty_like(f)
M.rhs(f, b)
out = []
for _ in range(2):
    M.ax(f, y)
    out += [y.clone(), (M.cg_solve(b, x, 0.0, 20), x.clone())[1], (M.cg_solve(b, x, 1e-6, 500), x.clone())[1]]
torch.cuda.synchronize()
assert all(torch.equal(a, c) for a, c in zip(out[:3], out[3:]))
torch.save([t.cpu() for t in out], sys.argv[2])
"""


def test_one_form_at_a_time(semlib, tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = {}
    for how in ("both", "one"):
        path = str(tmp_path / how)
        subprocess.run([sys.executable, "-c", CHILD, how, path], cwd=root, check=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=root))
        got[how] = torch.load(path)
    assert all(torch.equal(a, b) for a, b in zip(got["both"], got["one"]))


MIXED = """
import sys
import torch
from paper_2606_12650_gb300 import Mesh, sem
from paper_2606_12650_gb300.inputs import box_vertices, normal_field
nL = 10 ** 3 * 512
if sys.argv[1] == "one":
    sem.init(["--device=0", "--hbm-budget=%.9f" % (nL * (96 + 28 + 48 + 30) / 1e9)])   # 28: BF16 factors and FP32 vectors
else:
    sem.init(["--device=0"])
torch.cuda.set_stream(sem.stream())
M = Mesh(10, 10, 10, 7, box_vertices(10, 10, 10, 0.05, seed=1))
f = torch.from_numpy(normal_field(M.nL, 3)).cuda()
b, x = torch.empty_like(f), torch.empty_like(f)
M.rhs(f, b)
out = []
for _ in range(2):
    M.cg_solve(b, x, 0.0, 20)
    out.append(x.clone())
    out.append(torch.tensor(M.cg_mixed(b, x, 1e-9)))      # its residual makes the integer form, in the other's place, between inner solves
    out.append(x.clone())
torch.cuda.synchronize()
torch.save([t.cpu() for t in out], sys.argv[2])
"""


def test_the_form_changes_within_a_mixed_solve(semlib, tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = {}
    for how in ("both", "one"):
        path = str(tmp_path / how)
        subprocess.run([sys.executable, "-c", MIXED, how, path], cwd=root, check=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=root))
        got[how] = torch.load(path)
    assert all(torch.equal(a, b) for a, b in zip(got["both"], got["one"]))
