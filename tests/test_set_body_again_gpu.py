"""Bodies set one after the other in a context: growing, shrinking and of the same
size (the ghost band then keeps its memory), each against a fresh context, bit for
bit, with the same device bytes."""
import numpy as np
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim", [2, 3])
def test_bodies_in_turn(dim, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    make = wl.circle if dim == 2 else wl.sphere
    bodies = [make(r) for r in (0.7, 0.9, 0.85, 0.85, 0.2, 0.9)] + [{"kind": "none"}, make(0.6)]

    def case(body):
        n, nv = (64, 24) if dim == 2 else (16, 10)
        return wl._case(dim, n, 2.0, nv, 4.5, 0.2, 0.3, body, precision=precision)

    stream = torch.cuda.Stream()
    s = ibdvm.Solver(case({"kind": "none"}), stream=stream.cuda_stream)
    f0 = s.get_f() * (1.0 + 0.05 * np.random.default_rng(1).uniform(-1.0, 1.0, size=s.shape()))
    for body in bodies:
        s.set_body(body)
        fresh = ibdvm.Solver(case(body), stream=stream.cuda_stream)
        out = []
        for x in (s, fresh):
            x.set_f(f0)
            r = x.step(4)
            W, q, t = x.moments()
            fluid = t == 0
            out.append((x.get_f()[fluid], W[fluid], q[fluid], [r], np.concatenate([np.ravel(v) for v in x.step_forces()])))
            x.refresh_info()
        for a, b in zip(*out):
            np.testing.assert_array_equal(a, b)
        assert s.info.device_bytes == fresh.info.device_bytes
        fresh.close()
    s.close()
