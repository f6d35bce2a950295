"""The work items of a 2D batch without a tiling: whole columns where the members
have many, ranges of rows where they have few, and the tuner tries that choice."""
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def items(b):
    b.step(2)
    return b.tiling()["nitems"]


@pytest.mark.parametrize("members,whole", [(1, False), (10, True)])
def test_items_by_the_number_of_columns(members, whole):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # 100 strips of 8 columns, 4 velocity chunks: 400 columns of 96 rows a member
    c = wl._case(2, [800, 96], 2.0, 16, 4.5, 0.4, 0.3, {"kind": "none"}, precision="mixed")
    stream = torch.cuda.Stream()
    b = ibdvm.Batch(stream=stream.cuda_stream)
    solvers = [ibdvm.Solver(c, stream=stream.cuda_stream) for _ in range(members)]
    for s in solvers:
        b.add(s)
    auto = items(b)
    b.tune(2)
    tuned = b.tiling()
    b.set_tiling(0)
    columns = items(b)
    assert columns == 400 * members and auto == (1 if whole else 2) * columns
    assert tuned["rows"] in (0, 16, 32, 128)
    b.close()
    for s in solvers:
        s.close()
