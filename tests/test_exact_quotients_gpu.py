"""Moments whose sums and quotients are whole numbers come out exact.

f is symmetric about the node (1, 0) on nine unit-weight nodes, and its values
are whole numbers, so the sums, the bulk velocity (1, 0) and the heat flux 0
have no rounding at all, whatever the order of the sums: W and q equal them bit
for bit.  The densities include values n for which n times the rounded 1 / n is
not 1 (49, 98, 103, 107, 161)."""
import numpy as np
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_whole_number_state(precision):
    pytest.importorskip("torch")
    case = wl._case(2, [8, 8], 2.0, 9, 4.0, 0.5, 0.1, {"kind": "none"}, dt=1e-6, precision=precision)
    s = ibdvm.Solver(case)
    f = np.zeros(s.shape())
    rho = np.resize([49, 98, 103, 107, 161, 3, 10, 64], s.ncell)
    node = lambda x, y: (x + 4) + 9 * (y + 4)
    rest = rho.copy()
    for x, y, n in ((0, 0, 1), (1, 1, 2), (0, 1, 3), (0, -1, 5)):  # n at (x, y) and at its mirror (2 - x, -y)
        n = np.where(rest > 2 * n, n, 0)
        f[:, node(x, y), 0] += n
        f[:, node(2 - x, -y), 0] += n
        rest = rest - 2 * n
    f[:, node(1, 0), 0] += rest
    s.set_f(f)
    W, q, _ = s.moments()
    xi = np.array([[x, y] for y in range(-4, 5) for x in range(-4, 5)], dtype=float)
    np.testing.assert_array_equal(W[:, 0], rho)
    np.testing.assert_array_equal(W[:, 1], rho)
    np.testing.assert_array_equal(W[:, 2], np.zeros(s.ncell))
    np.testing.assert_array_equal(W[:, 3], 0.5 * (f[:, :, 0] @ (xi * xi).sum(1)))
    np.testing.assert_array_equal(q, np.zeros((s.ncell, 2)))
    s.close()
