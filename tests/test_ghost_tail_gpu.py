"""Ghost values of the FP64 path in the tail of a cold gas before a hot wall.

A velocity whose box lies wholly on the incident side keeps the incident value,
however much larger the reflected Maxwellian is there (25 orders and more here).
The box measure is 49/256, whose product with its rounded reciprocal is not 1.
Entry by entry against the oracle, relative to the entry before or after the
step: the operations of the step are on values of that size (neighbouring cells
differ by 10 %), so the entries agree to a few hundred roundings (1e-12, which
allows for cancellation in the extrapolations).  Boxes that the wall plane cuts
are left out: their measures are two codes' own, and so are their roundings."""
import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_incident_tail_before_a_hot_wall():
    pytest.importorskip("torch")
    case = wl._case(2, [24, 24], 2.0, 20, 4.15625, 0.5, 0.1, dict(wl.circle(0.7), Tw=4.0), T_inf=0.25)
    o = oracle.OracleCase(case)
    _, w = o.velocities()
    assert np.any(w * (1.0 / w) != 1.0) and np.any(o.cut_table() == w)
    f0 = o.get_f() * (1.0 + 0.1 * np.random.default_rng(5).uniform(-1.0, 1.0, size=o.shape()))
    g = ibdvm.Solver(case)
    g.set_f(f0)
    o.set_f(f0)
    g.step(1)
    o.step(1)
    fl = o.cell_types() == oracle.FLUID
    fg, fo = g.get_f()[fl], o.get_f()[fl]
    g.close()
    whole = np.ones((o.ncell, o.nvel), dtype=bool)  # no reflected share in a link of the cell
    for donor, wg in zip(o.links()["donor"], o.cut_table()):
        whole[donor] &= wg == w
    size = np.maximum(f0[fl], np.abs(fo))
    assert size.min() < 1e-25 * size.max()
    assert np.max((np.abs(fg - fo) / size)[whole[fl]]) < 1e-12
