"""The ghost band and the surface force, whose links are split over clusters of
blocks: velocity counts that leave some of a cluster's blocks empty or ragged,
accommodation coefficients with and without the specular part, one link to many,
against the oracle (FP64 1e-11 relative; FP32 storage 1e-5, the path's
tolerance; the force ten times that, a sum of differences)."""
import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 1e-5)])
@pytest.mark.parametrize("accom", [1.0, 0.6, 0.0])
@pytest.mark.parametrize("dim,n,nv", [(2, 12, 3), (2, 24, 9), (2, 31, 33), (3, 8, 4), (3, 8, 12)])
def test_links_against_the_oracle(dim, n, nv, accom, precision, tol):
    pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    body = wl.circle(0.61, center=(0.1, -0.05), accom=accom, Tw=1.2) if dim == 2 else \
        wl.sphere(0.62, center=(0.1, -0.05, 0.07), accom=accom, Tw=1.2)
    case = wl._case(dim, n, 1.5, nv, 3.5, 0.2, 0.4, body, precision=precision)
    g, o = ibdvm.Solver(case), oracle.OracleCase(case)
    f0 = o.get_f() * (1.0 + 0.2 * np.random.default_rng(7).uniform(-1.0, 1.0, size=o.shape()))
    g.set_f(f0)
    o.set_f(f0)
    assert g.nlink > 0
    gb, ob = g.ghost_band(), o.ghost_band()
    for k in ("fiw", "fstarw", "fstargc"):
        assert np.abs(gb[k] - ob[k]).max() < tol * np.abs(ob[k]).max(), k
    if accom > 0.0:
        np.testing.assert_allclose(gb["rhow"], ob["rhow"], rtol=10 * tol)
    for _ in range(2):  # the counter of finished blocks starts over
        F, Q, _, _ = g.forces()
        Fo, Qo, _, _ = o.forces()
        scale = max(np.abs(Fo).max(), abs(Qo))
        assert np.abs(F - Fo).max() < 10 * tol * scale and abs(Q - Qo) < 10 * tol * scale
    g.close()
