"""The work items of a 2D batch whose tiling was not set: about 64 rows each.

The row ranges change no cell's arithmetic, so the states, residuals and forces
are bit for bit those of whole columns, at the row counts where the number of
ranges changes (95 / 96, 159 / 160) and where they are uneven (161)."""
import numpy as np
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [9, 95, 96, 159, 160, 161])
def test_untiled_batch_matches_whole_columns(ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = wl.small_2d("circle", n=19, nv=8, Ma=0.3, precision="mixed", Kn=0.4)
    c["n"] = [19, ny]
    c["lo"], c["hi"] = [-1.5, -0.08 * ny], [1.5, 0.08 * ny]
    stream = torch.cuda.Stream()
    out = []
    for whole in (True, False):
        m = ibdvm.Solver(c, stream=stream.cuda_stream)
        b = ibdvm.Batch(stream=stream.cuda_stream)
        b.add(m)
        if whole:
            b.set_tiling(0, 0)
        r, st = b.step(3)
        assert list(st) == [0] and b.tiling()["rows"] == 0
        out.append((m.get_f(), list(r), b.forces(), b.tiling()["nitems"]))
        b.close()
        m.close()
    (f0, r0, F0, n0), (f1, r1, F1, n1) = out
    np.testing.assert_array_equal(f0, f1)
    assert r0 == r1
    for a, b in zip(F0, F1):
        np.testing.assert_array_equal(a, b)
    assert n1 == n0 * max(1, (ny + 32) // 64)
