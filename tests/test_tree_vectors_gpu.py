"""The FP32 tree sweep's 16-byte vectors where orthants end inside them: odd and
uneven velocity counts per axis (every octant of another size, vectors that hold
two orthants or end in padding), quadtrees and octrees, against the oracle
within 1e-5 on f, the mixed path's tolerance; and that padding keeps zeros."""
import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,nv", [(2, (13, 11)), (2, (16, 9)), (2, (33, 14)), (3, (7, 5, 9)), (3, (9, 8, 7)),
                                    (3, (6, 11, 8))])
def test_straddling_vectors(dim, nv):
    pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    case = (wl.tree_case(12, 2, Ma=0.4, Kn=0.3, precision="mixed") if dim == 2 else
            wl.tree_case_3d(6, 2, Ma=0.4, Kn=0.3, precision="mixed"))
    case["nv"] = list(nv)
    g, o = ibdvm.Solver(case), oracle.OracleTree(case)
    f0 = o.get_f() * (1.0 + 0.1 * np.random.default_rng(4).uniform(-1.0, 1.0, size=o.shape()))
    g.set_f(f0)
    o.set_f(f0)
    g.step(3)
    o.step(3)
    fo = o.get_f()
    assert np.abs(g.get_f() - fo).max() < 1e-5 * np.abs(fo).max()
    raw = np.zeros(g.native_shape(), dtype=np.float32)
    g.get_f_native(raw.ctypes.data, raw.nbytes)
    pad = np.setdiff1d(np.arange(g.nvel_padded), g.velocity_positions())
    assert not raw[:, pad].any()
    g.close()
