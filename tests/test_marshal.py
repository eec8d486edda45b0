"""The argument records that run() passes are those of the general marshalling,
byte for byte, for every kind of argument (CPU)."""
import numpy as np
import pytest

from paper_2606_12650_gb300 import sem

torch = pytest.importorskip("torch")


def test_records_match():
    host = np.arange(4.0)
    args = [0, 7, -3, 2 ** 63 - 1, -2 ** 63, 1.5, -0.0, float("inf"), None, sem.OutInt(), sem.OutDouble(),
            sem.HostArray(host), sem.HostPtr(4096), sem.DevicePtr(8192), host, torch.arange(3.0),
            torch.nn.Parameter(torch.zeros(2))]
    for n in range(len(args) + 1):
        recs = (sem.SemArg * max(n, 1))(*[sem._marshal(a) for a in args[:n]])
        assert sem._pack(args[:n]) == bytes(recs)[:16 * n]


def test_what_was_refused_stays_refused():
    for bad, error in ((True, TypeError), ("x", TypeError), (np.zeros((4, 4)).T[1:], ValueError),
                       (torch.zeros(4, 4).T, ValueError)):
        with pytest.raises(error):
            sem._marshal(bad)
        with pytest.raises(error):
            sem._pack([1, bad])
