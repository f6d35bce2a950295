"""Roundings of one FP32 step on trees.

Against the FP64 step from the same FP32 values, at a CFL number of 1/64: the
increments of transport and relaxation are below 1/64 of f (neighbours differ
by 10 %), so their own roundings (about eight of 2^-24 relative) move f by less
than a quarter of a unit in its last place (velocities up to 3, so that products of differences
stay normal FP32 numbers); f^{n+1} itself is rounded once, half
a unit.  With the FP32 Maxwellian parameters' share (dt / tau of 1e-3 times some
hundred roundings) less than one unit in all.

The equilibrium of an octree: a state of 24 velocities with c^2 = 3/2 has
rho = 3, U = 0, T = 1 and q = 0 exactly, so where f is zero the step leaves
dt/tau rho / pi^1.5 exp(-c^2), and the ratio to the value at c = 0 errs by the
exponential (two units) and two products on each side: below 5 2^-23."""
import numpy as np
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
def test_one_rounding_at_the_size_of_f(dim):
    pytest.importorskip("torch")
    out = {}
    for precision in ("fp64", "mixed"):
        make = wl.tree_case if dim == 2 else wl.tree_case_3d
        case = make(12 if dim == 2 else 6, 2, V=3.0, Ma=0.4, Kn=0.3, precision=precision)
        case["cfl"] = 1.0 / 64.0
        s = ibdvm.Solver(case)
        f0 = s.get_f().astype(np.float32).astype(np.float64)
        f0 = f0[:1] * (1.0 + 0.1 * np.random.default_rng(2).uniform(-1.0, 1.0, size=f0.shape))
        s.set_f(f0.astype(np.float32).astype(np.float64))
        s.step(1)
        out[precision] = s.get_f()
        s.close()
    unit = np.spacing(np.abs(out["fp64"]).astype(np.float32)).astype(np.float64)
    assert np.max(np.abs(out["mixed"] - out["fp64"]) / unit) < 1.0


def test_octree_equilibrium_in_the_tail():
    pytest.importorskip("torch")
    case = wl.tree_case_3d(6, 1, Ma=0.0, Kn=0.3, precision="mixed")
    case.update(nv=[17] * 3, vlo=[-4.0] * 3, vhi=[4.0] * 3)
    s = ibdvm.Solver(case)
    x = -4.0 + 0.5 * np.arange(17)
    xi = np.stack(np.meshgrid(x, x, x, indexing="ij")[::-1], axis=-1).reshape(-1, 3)
    c2 = (xi * xi).sum(1)
    on = (c2 == 1.5) & (np.abs(xi).min(1) == 0.5)
    assert on.sum() == 24
    f = np.zeros(s.shape())
    f[:, on] = 1.0
    s.set_f(f)
    s.step(1)
    f = s.get_f()[:, :, 0]
    s.close()
    h = (case["hi"][0] - case["lo"][0]) / case["n"][0]
    inner = np.all(np.abs(wl.tree_centres(case)) < case["hi"][0] - 2.0 * h, axis=1)
    assert inner.sum() >= 8
    rest = f[inner][:, c2 == 0.0]
    np.testing.assert_allclose(f[inner][:, ~on] / rest, np.tile(np.exp(-c2[~on]), (inner.sum(), 1)), rtol=5 * 2.0 ** -23)
