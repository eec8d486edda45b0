"""The exchange between the blocks of a one-kernel solve gives up in time.

40 blocks take part in the exchange of 41: the second group's leader waits for
a slot that nobody fills, the others for the leader's.  Every wait ends after
its limit, the next sem_sync names the exchange, and solves after it, in one
kernel and of the same problem, are those before it bit for bit.
"""
import pytest

from paper_2606_12650_gb300.inputs import box_vertices, normal_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_wait_runs_out_and_solves_go_on(semlib):
    from paper_2606_12650_gb300 import Mesh, sem
    M = Mesh(5, 4, 3, 5, box_vertices(5, 4, 3, 0.05, seed=1))      # 60 elements: two groups
    f = torch.from_numpy(normal_field(M.nL, 3)).cuda()
    b, xs = torch.empty_like(f), []
    M.rhs(f, b)
    for probe in (False, True):
        if probe:
            sem.run("exchange_probe", 100000)
            with pytest.raises(sem.SemError) as e:
                sem.sync()
            assert e.value.code == sem.SEM_ETIMEDOUT and "exchange" in e.value.message
            sem.sync()
        x = torch.empty_like(b)
        it, res = M.cg_solve(b, x, 1e-8, 1000)
        xs.append((it, res, x))
    assert xs[0][:2] == xs[1][:2] and torch.equal(xs[0][2], xs[1][2])
    sem.run("exchange_probe", 100000)
    with pytest.raises(sem.SemError) as e:                          # a solve's own poll sees it too
        M.pcg_solve(b, torch.empty_like(b), 1e-8, 1000)
    assert e.value.code == sem.SEM_ETIMEDOUT
    M.free()


def test_limits(semlib):
    from paper_2606_12650_gb300 import sem
    with pytest.raises(sem.SemError) as e:
        sem.run("exchange_probe", 10)
    assert e.value.code == sem.SEM_EARG
