"""The launches that kernel_times reports for the ghost band are those that run:
the slope kernel and the band kernel, or the band kernel alone where every link
extrapolates linearly (upwind = 3 reads no slopes), in a solver and in a batch."""
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("upwind,batch,want", [((1,), False, 2), ((3,), False, 1), ((1,), True, 2), ((3,), True, 1),
                                               ((3, 1), True, 2)])
def test_ghost_band_launches(upwind, batch, want):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stream = torch.cuda.Stream()
    solvers = [ibdvm.Solver(wl.small_2d("circle", n=24, nv=8, precision="mixed", upwind=u), stream=stream.cuda_stream)
               for u in upwind]
    o = solvers[0]
    if batch:
        o = ibdvm.Batch(stream=stream.cuda_stream)
        for s in solvers:
            o.add(s)
    o.step(1)
    o.reset_kernel_times()
    o.step(1)
    assert o.kernel_times()["ghost_band"][1] == want
    if batch:
        o.close()
    for s in solvers:
        s.close()
