"""The halo kernel of diffuse domain walls: blocks of one boundary cell on
small faces, blocks of four that do not divide a large one, velocity grids with
a zero component, walls on some faces only and at different temperatures.
Tolerances as the other parity tests: 1e-11 in FP64, 1e-5 in the mixed path
(FP32 storage: 170 roundings of 6e-8)."""
import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,nv,faces", [
    ((5, 7), 9, (0, 1, 2, 3)),
    ((6, 4), 8, (1, 2)),
    ((9, 11), 7, (3,)),
    ((5, 6, 7), 6, (0, 1, 2, 3, 4, 5)),
    ((4, 5, 5), 7, (2, 4, 5)),
    ((701, 6), 6, (2, 3)),
])
def test_wall_halo_against_the_oracle(n, nv, faces, precision):
    pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    dim = len(n)
    walls = [None] * 6
    for i in faces:
        walls[i] = {"Tw": 0.8 + 0.1 * i, "Uw": [0.1 if a != i // 2 else 0.0 for a in range(dim)] + [0.0] * (3 - dim)}
    case = wl._case(dim, list(n), ([0.0] * dim, [1.0] * dim), nv, 4.5, 0.2, 0.0, {"kind": "none"},
                    precision=precision, domain_walls=walls)
    g, o = ibdvm.Solver(case), oracle.OracleCase(case)
    f0 = o.get_f() * (1.0 + 0.3 * np.random.default_rng(5).uniform(-1.0, 1.0, size=o.shape()))
    g.set_f(f0)
    o.set_f(f0)
    g.step(3)
    o.step(3)
    fg, fo = g.get_f(), o.get_f()
    g.close()
    assert np.abs(fg - fo).max() < (1e-11 if precision == "fp64" else 1e-5) * np.abs(fo).max()
