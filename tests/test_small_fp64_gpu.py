"""FP64 cases on the smallest grids and on grids of four columns take the direct
sweep (one launch), the others the sweep that forms every face once (a table
launch and the sweep): on both sides of the rule's edges (152 blocks of four cells
and 64 velocities; four columns in 2D), with a body and walls, against the oracle
within 1e-11, the FP64 path's tolerance."""
import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,nv,kind,launches", [
    (2, (4, 4), 24, "none", 1), (2, (19, 32), 8, "circle", 1), (2, (19, 33), 8, "circle", 2), (2, (12, 12), 16, "walls", 1),
    (2, (12, 13), 16, "walls", 2), (2, (4, 90), 17, "walls", 1), (2, (5, 90), 17, "walls", 2), (3, (4, 4, 4), 6, "none", 1),
    (3, (8, 8, 9), 4, "sphere", 1), (3, (8, 8, 10), 4, "sphere", 2), (3, (5, 4, 4), 9, "walls", 2)])
def test_both_sides_of_the_rule(dim, n, nv, kind, launches):
    pytest.importorskip("torch")
    body = {"circle": wl.circle(0.55), "sphere": wl.sphere(0.9)}.get(kind, {"kind": "none"})
    kw = {"domain_walls": wl.box_walls(dim, 1.1, lid=(0.2, 0.0, 0.0)[:dim])} if kind == "walls" else {}
    case = wl._case(dim, list(n), 2.0, nv, 4.5, 0.3, 0.3, body, **kw)
    g, o = ibdvm.Solver(case), oracle.OracleCase(case)
    f0 = o.get_f() * (1.0 + 0.2 * np.random.default_rng(8).uniform(-1.0, 1.0, size=o.shape()))
    g.set_f(f0)
    o.set_f(f0)
    g.reset_kernel_times()
    rg, ro = g.step(2), o.step(2)
    assert g.kernel_times()["sweep"][1] == 2 * launches
    fl = o.cell_types() == oracle.FLUID
    fg, fo = g.get_f()[fl], o.get_f()[fl]
    (Wg, qg, _), (Wo, qo) = g.moments(), o.moments()
    g.close()
    assert np.abs(fg - fo).max() < 1e-11 * np.abs(fo).max()
    assert np.abs(Wg[fl] - Wo[fl]).max() < 1e-11 * np.abs(Wo[fl]).max()
    assert np.abs(qg[fl] - qo[fl]).max() < 1e-11 * np.abs(Wo[fl]).max()
    assert rg == pytest.approx(ro, rel=1e-9)
