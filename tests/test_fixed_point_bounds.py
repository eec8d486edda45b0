"""The integer sums of the fixed-point operator stay within 64 bits (no GPU).

The scales follow sem_ax_fx.cuh: |X| < 2^60, |G| < 2^62, the coefficients of D
and D^T times the largest 2^k for which a row's cross terms stay below 2^63.
With every factor at its bound and every sign aligned (more than any mesh
gives), |U| <= R c for the row sums R of |D|, |W| <= (R_i + R_j + R_k) c / 4, and
|Y| follows by |D^T|.  Of <p, y> a thread's cross terms (at N = 9 of five nodes at
a time) and its own sum must fit; the element's sum passes 2^63 at high
orders, so the upper 20 bits of the threads' sums are added apart.
"""
import numpy as np
import pytest


def _gll_derivative(N):
    P = np.polynomial.legendre.Legendre.basis(N)
    xi = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    d = xi[:, None] - xi[None, :] + np.eye(N + 1)
    lam = 1.0 / d.prod(axis=1)
    D = lam[None, :] / lam[:, None] / d
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, -D.sum(axis=1))
    return D


def _scale(M, ubound):
    n = len(M)
    H, odd = n // 2, n % 2
    e = 0.5 * (M[:H, :H] + M[:H, ::-1][:, :H])
    o = 0.5 * (M[:H + odd, :H] - M[:H + odd, ::-1][:, :H])
    mid = np.abs(M[:H, H]) if odd else np.zeros(H)
    big = max(np.abs(e).max(), np.abs(o).max(), mid.max())
    row = max((np.abs(e).sum(axis=1) + mid).max(), np.abs(o).sum(axis=1).max())
    uh = (2 * H * ubound + odd * ubound) / 2.0 ** 32 + 2 * H + 2
    k = 0
    while big * 2.0 ** (k + 1) < 2.0 ** 63 - 2.0 ** 32 and (row * 2.0 ** (k + 1) / 2.0 ** 32 + uh) * 2.0 ** 31 < 2.0 ** 63:
        k += 1
    return k


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_sums_fit(N):
    n = N + 1
    D = _gll_derivative(N)
    A, R = np.abs(D), np.abs(D).sum(axis=1)
    k1 = _scale(D, 2.0 ** 60)
    U = R.max() * 2.0 ** (k1 - 4)
    k2 = _scale(D.T, 3 * 2.0 ** -2 * U)
    W = (R[:, None, None] + R[None, :, None] + R[None, None, :]) * 2.0 ** (k1 - 4) / 4
    Y = 2.0 ** (k2 - 64) * (np.einsum("li,lbc->ibc", A, W) + np.einsum("lj,alc->ajc", A, W) + np.einsum("lk,abl->abk", A, W))
    assert Y.max() < 2.0 ** 62                                   # also times the headroom shift of the last cut
    cross = lambda y: 2.0 ** 59 + 2.0 ** 31 * (y / 2.0 ** 32 + 1)   # |xh yl| + |xl yh| of a node
    line = Y.reshape(n * n, n)                                   # a thread's nodes (the map is symmetric in the directions)
    per = 5 if n == 10 else n
    for first in range(0, n, per):
        assert cross(line[:, first:first + per]).sum(axis=1).max() + 2.0 ** 31 < 2.0 ** 63
    thread = (2.0 ** 60 * line / 2.0 ** 64 + cross(line) / 2.0 ** 32).sum(axis=1)
    assert thread.max() < 2.0 ** 63
    # fx_bound's form of the element's sum, all factors at their bound (|g| = 2)
    S = 2 * ((R[:, None, None] + R[None, :, None] + R[None, None, :]) ** 2).sum()
    np.testing.assert_allclose(2.0 ** 60 * Y.sum() / 2.0 ** 64, 2.0 ** (k1 + k2 - 75) * S, rtol=1e-12)
    assert 2.0 ** (k1 + k2 - 75) * S < 2.0 ** (62 + 8)           # eight bits less are enough
    # the rest of an element's sum: the cross terms' upper halves
    assert (0.99 * 2.0 ** 62 + n ** 3 * cross(Y.max()) / 2.0 ** 32) < 2.0 ** 63
