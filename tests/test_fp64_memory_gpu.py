"""FP64 cases on a device with little memory left: the sweep's tables take what the
rest of the case leaves, in slabs of rows, and give it back to a body's ghost band
and to wall halos.  The results are those of the same case with room to spare, bit
for bit: rows are swept by the same operations whatever their slab.

The test fills the device, so it does not run beside others (pytest-xdist)."""
import gc
import os

import numpy as np
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif("PYTEST_XDIST_WORKER" in os.environ, reason="fills the device memory")]

MB = 1 << 20


@pytest.fixture()
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.collect()
    torch.cuda.empty_cache()
    yield torch
    gc.collect()
    torch.cuda.empty_cache()


def free_bytes(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def fill(torch, spare):
    """All of the device's free memory but about `spare` bytes."""
    return torch.empty(max(free_bytes(torch) - int(spare), 0), dtype=torch.uint8, device="cuda")


def case(dim):
    walls = wl.box_walls(dim, 1.1, lid=(0.2, 0.0, 0.0)[:dim])
    if dim == 2:  # 300 x 800 cells: tables of 230 MB, 0.288 MB a row
        c = wl._case(2, [300, 800], 4.0, 12, 4.5, 0.2, 0.3, wl.circle(1.5), domain_walls=walls)
    else:  # 64 x 64 x 48 cells: tables of 132 MB
        c = wl._case(3, [64, 64, 48], 2.0, 6, 4.5, 0.2, 0.3, wl.sphere(1.7), domain_walls=walls)
    other = 4 * sum(c["nv"][1:])
    table = 8 * int(np.prod(c["n"])) * (6 * c["nv"][0] + other)
    return c, table


def place(s, c):
    s.set_body(c["body"])
    s.set_domain(c["domain_walls"])


def result(s, f0):
    s.set_f(f0)
    s.reset_kernel_times()
    res = s.step(3)
    n = s.kernel_times()["sweep"][1] // 3
    f, (W, q, _) = s.get_f(), s.moments()
    return (f, W, q, np.array([res]), np.concatenate([np.ravel(x) for x in s.step_forces()])), n


def measure(torch, dim):
    """The case, the same without body and walls, the bytes that the bare case takes
    beside its tables and that body and walls add, a state and its result."""
    c, table = case(dim)
    bare = dict(c, body={"kind": "none"}, domain_walls=None)
    free = [free_bytes(torch)]
    s = ibdvm.Solver(bare)
    free.append(free_bytes(torch))
    place(s, c)
    free.append(free_bytes(torch))
    f0 = s.get_f() * (1.0 + 0.1 * np.random.default_rng(3).uniform(-1.0, 1.0, size=s.shape()))
    want, launches = result(s, f0)
    s.close()
    assert launches == 2 and free[1] - free[2] > 8 * MB
    return c, bare, free[0] - free[1] - table, free[1] - free[2], f0, want


def same(s, f0, want):
    got, launches = result(s, f0)
    assert launches > 2
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


def test_tables_leave_room_for_the_body(torch):
    c, bare, rest, added, f0, want = measure(torch, 3)
    block = fill(torch, rest + added + 16 * MB)
    s = ibdvm.Solver(bare)
    try:
        place(s, c)
        del block
        torch.cuda.empty_cache()
        same(s, f0, want)
    finally:
        s.close()


@pytest.mark.parametrize("dim", [2, 3])
def test_tables_make_room_for_the_body(torch, dim):
    c, bare, _, added, f0, want = measure(torch, dim)
    s = ibdvm.Solver(bare)
    block = fill(torch, added // 2)
    try:
        place(s, c)
        del block
        torch.cuda.empty_cache()
        same(s, f0, want)
    finally:
        s.close()
