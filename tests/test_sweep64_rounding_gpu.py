"""Roundings of the FP64 sweep against extended precision.

f: at a CFL number of 1/64 the increments of transport and relaxation are below
1/64 of f's size (neighbours differ by 10 %), so their own roundings (about ten of
2^-53 relative) move f by less than a third of a unit in its last place; f^{n+1}
itself is rounded once, half a unit: less than one unit in all.  Interior cells,
whose stencil holds no halo.

The density against the sum of the returned f (weights that are powers of two, so
that both take the same ones): a group of up to eight
velocities, the four of a batch and its factor make some eleven roundings, each
0.3 units rms of the batch's share; those of 40 batches average out to below a
fifth of a unit, the compensated sums over batches and chunks and the last
rounding add about half a unit: 0.6 rms, below three units everywhere (five
standard deviations)."""
import numpy as np
import pytest

from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def one_step(f, xi, w, dt, h, mu0, omega, Pr):
    """f^{n+1} of the interior cells in extended precision (f[z, y, x][k][c], from
    the doubles the library holds)."""
    dim = f.ndim - 2
    m = f[..., 0] * w
    rho = m.sum(-1)
    U = [(m * xi[:, a]).sum(-1) / rho for a in range(dim)]
    c = [xi[:, a] - U[a][..., None] for a in range(dim)]
    c2 = sum(v * v for v in c)
    e = c2 * m + (f[..., 1] * w if dim == 2 else 0)
    T = LD(2) / 3 * e.sum(-1) / rho
    q = [(v * e).sum(-1) / 2 for v in c]
    corr = (4 * (1 - LD(Pr)) / (5 * rho * T * T))[..., None] * sum(v * k[..., None] for v, k in zip(c, q))
    g = (rho / (PI * T) ** (LD(dim) / 2 if dim == 3 else LD(1)))[..., None] * np.exp(-c2 / T[..., None])
    t = 2 * c2 / T[..., None]
    eq = (np.stack([g * (1 + corr * (t - 4)), T[..., None] / 2 * g * (1 + corr * (t - 2))], -1) if dim == 2 else
          (g * (1 + corr * (t - 5)))[..., None])
    new = f + (LD(dt) * rho * T / 2 / (LD(mu0) * T ** LD(omega)))[..., None, None] * (eq - f)
    for a in range(dim):
        ax = dim - 1 - a
        d = np.diff(f, axis=ax)
        lo, hi = np.take(d, range(d.shape[ax] - 1), ax), np.take(d, range(1, d.shape[ax]), ax)
        p = lo * hi
        half = np.where(p > 0, p / np.where(p > 0, lo + hi, 1), 0)  # cells 1 .. n - 2
        mid = np.take(f, range(1, f.shape[ax] - 1), ax)
        right, left = mid + half, mid - half
        x = xi[:, a, None]
        cut = lambda v, s: np.take(v, range(1 + s, v.shape[ax] - 1 + s), ax)
        flux = np.where(x > 0, cut(right, 0) - cut(right, -1), cut(left, 1) - cut(left, 0)) * x / LD(h[a])
        np.moveaxis(new, ax, 0)[2:-2] -= LD(dt) * np.moveaxis(flux, ax, 0)
    return new[(slice(2, -2),) * dim]


@pytest.mark.parametrize("dim,n,nv", [(2, (21, 18), 17), (3, (9, 7, 8), 10)])
def test_one_rounding_at_the_size_of_f(dim, n, nv):
    pytest.importorskip("torch")
    case = wl._case(dim, list(n), 2.0, nv, 3.0, 0.3, 0.4, {"kind": "none"}, cfl=1.0 / 64.0)
    s = ibdvm.Solver(case)
    f0 = s.get_f()
    f0 = f0 * (1.0 + 0.1 * np.random.default_rng(6).uniform(-1.0, 1.0, size=f0.shape))
    s.set_f(f0)
    s.step(1)
    f = s.get_f()
    xi, w = s.geometry().velocities()
    h = [(case["hi"][a] - case["lo"][a]) / case["n"][a] for a in range(dim)]
    al, om = case["alpha_vhs"], case["omega_vhs"]
    mu0 = 5 * (al + 1) * (al + 2) * np.sqrt(PI) / (4 * al * (5 - 2 * om) * (7 - 2 * om)) * case["Kn"]
    shape = tuple(n[::-1]) + f.shape[1:]
    want = one_step(f0.reshape(shape).astype(LD), xi.astype(LD), w.astype(LD), s.info.dt, h, mu0, om, case["Pr"])
    s.close()
    got = f.reshape(shape)[(slice(2, -2),) * dim]
    assert float(np.max(np.abs(got - want) / np.spacing(np.abs(got)))) < 1.0


@pytest.mark.parametrize("dim,n,nv", [(2, (24, 20), 33), (3, (7, 6, 6), 9)])
def test_density_of_the_returned_state(dim, n, nv):
    pytest.importorskip("torch")
    s = ibdvm.Solver(wl._case(dim, list(n), 2.0, nv, 4.0, 0.3, 0.4, {"kind": "none"}))
    f0 = s.get_f()
    s.set_f(f0 * (1.0 + 0.1 * np.random.default_rng(7).uniform(-1.0, 1.0, size=f0.shape)))
    s.step(1)
    W, _, _ = s.moments()
    _, w = s.geometry().velocities()
    rho = (s.get_f()[:, :, 0].astype(LD) * w).sum(1)
    s.close()
    assert float(np.max(np.abs(W[:, 0] - rho) / rho)) < 3 * 2.0 ** -53
