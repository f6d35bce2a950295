"""Admission by the HBM budget: a second request is admitted beside the first where
both fit by a margin of 60 % of one (the estimate counts the partial sums of both
storage types, 30 % in 3D), for bodies of every kind; the bytes on the
device stay within the budget."""
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

BODIES = {"none": (2, {"kind": "none"}), "circle": (2, wl.circle(0.7)), "ellipse": (2, wl.ellipse(0.4, 1.8, 0.5)),
          "polygon": (2, wl.naca0012(2.5, 7.0, 60)), "sphere": (3, wl.sphere(0.7))}


def case(dim, body):
    return wl._case(dim, 96 if dim == 2 else 32, 2.0, 24 if dim == 2 else 12, 4.5, 0.2, 0.3, body, precision="mixed")


def serve(n, c, budget):
    s = ibdvm.Server(tol=0.0, max_steps=4, steps_per_round=2, hbm_budget=budget)
    ids = [s.submit(c) for _ in range(n)]
    while any(s.poll()[:2]):
        pass
    out = [s.result(i) for i in ids]
    s.close()
    return out


@pytest.mark.parametrize("kind", list(BODIES))
def test_two_requests_that_fit_run_together(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = case(*BODIES[kind])
    size = serve(1, c, 0)[0]["device_bytes"]
    budget = int(2.6 * size)
    a, b = serve(2, c, budget)
    assert b["t_admit"] < a["t_done"] and a["device_bytes"] + b["device_bytes"] <= budget
    a, b = serve(2, c, int(1.9 * size))
    assert b["t_admit"] >= a["t_done"]
