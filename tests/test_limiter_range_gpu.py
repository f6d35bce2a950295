"""The FP64 sweep's limiter quotient over the exponents of its arguments.

With a Knudsen number so large that nothing relaxes, the step is linear in the
scale of the state but for the limiter's product and quotient, which see f^2 and
f^2 / f: states scaled by 2^-480 to 2^400 (products from 2^-1000 to 2^820, inside the
normal numbers for all but the last digits of nearly equal cells) against the
oracle, which divides, entry by entry within 1e-12 (neighbours differ by 30 %)."""
import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,nv", [(2, (33, 18), 9), (3, (9, 7, 8), 7)])
@pytest.mark.parametrize("power", [-480, -300, -100, 0, 150, 400])
def test_scaled_states(dim, n, nv, power):
    pytest.importorskip("torch")
    case = wl._case(dim, list(n), 2.0, nv, 2.0, 2.0 ** 200 * 2.0 ** max(power, 0), 0.3, {"kind": "none"})
    g, o = ibdvm.Solver(case), oracle.OracleCase(case)
    f0 = o.get_f() * (1.0 + 0.3 * np.random.default_rng(9).uniform(-1.0, 1.0, size=o.shape())) * 2.0 ** power
    g.set_f(f0)
    o.set_f(f0)
    g.step(1)
    o.step(1)
    # cells whose stencils hold no halo (the freestream is not scaled)
    inner = np.ones(n[::-1], dtype=bool)
    for a in range(dim):
        np.moveaxis(inner, a, 0)[[0, 1, -2, -1]] = False
    fg, fo = g.get_f()[inner.ravel()], o.get_f()[inner.ravel()]
    g.close()
    assert fo.min() > 0.0
    assert np.max(np.abs(fg - fo) / fo) < 1e-12
