"""The FP64 sweep of uniform grids at the edges of its tiles (16 columns in 2D,
8 x 4 in 3D), of its velocity groups (eight nodes of one sign, pairs of rows in
2D) and of its slabs of rows, against the oracle within 1e-11 on f and W, the
FP64 path's tolerance."""
import os

import numpy as np
import pytest

import oracle
from paper_2512_20252_gb300 import ibdvm
from paper_2512_20252_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = 1e-11


def check(case, steps=2, seed=3, threads=1):
    pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    g, o = ibdvm.Solver(case), oracle.OracleCase(case, threads=threads)
    f0 = o.get_f() * (1.0 + 0.3 * np.random.default_rng(seed).uniform(-1.0, 1.0, size=o.shape()))
    g.set_f(f0)
    o.set_f(f0)
    rg, ro = g.step(steps), o.step(steps)
    fl = o.cell_types() == oracle.FLUID
    fg, fo = g.get_f()[fl], o.get_f()[fl]
    Wg, qg, _ = g.moments()
    Wo, qo = o.moments()
    g.close()
    assert np.abs(fg - fo).max() < TOL * np.abs(fo).max()
    assert np.abs(Wg[fl] - Wo[fl]).max() < TOL * np.abs(Wo[fl]).max()
    assert np.abs(qg[fl] - qo[fl]).max() < TOL * np.abs(Wo[fl]).max()
    assert rg == pytest.approx(ro, rel=1e-9)


@pytest.mark.parametrize("n", [(4, 4), (15, 33), (16, 5), (17, 40), (31, 6), (33, 16)])
@pytest.mark.parametrize("nv", [(2, 3), (9, 8), (16, 17), (18, 5)])
def test_tiles_and_groups_2d(n, nv):
    check(wl._case(2, list(n), 2.0, list(nv), 4.0, 0.2, 0.3, {"kind": "none"}))


@pytest.mark.parametrize("n", [(4, 4, 4), (7, 5, 17), (8, 4, 6), (9, 3 + 4, 5), (17, 9, 16)])
@pytest.mark.parametrize("nv", [(3, 2, 4), (8, 9, 5), (17, 4, 3)])
def test_tiles_and_groups_3d(n, nv):
    check(wl._case(3, list(n), 2.0, list(nv), 4.0, 0.2, 0.3, {"kind": "none"}))


@pytest.mark.parametrize("center", [(0.0, 0.0), (-1.9, 1.3), (0.1, -1.95), (1.97, 0.2)])
@pytest.mark.parametrize("walls", [False, True])
def test_bodies_across_tile_and_domain_edges_2d(center, walls):
    kw = {"domain_walls": wl.box_walls(2, 1.1, lid=(0.2, 0.0))} if walls else {}
    check(wl._case(2, [37, 35], 2.0, 10, 4.5, 0.1, 0.4, wl.circle(0.55, center=center), **kw), steps=3)


@pytest.mark.parametrize("center", [(0.0, 0.0, 0.0), (-1.4, 0.2, 1.5), (0.3, 1.6, -0.2)])
def test_bodies_across_tile_and_domain_edges_3d(center):
    check(wl._case(3, [13, 11, 12], 2.0, 7, 4.5, 0.1, 0.4, wl.sphere(0.8, center=center)), steps=3)


def test_one_signed_velocities():
    """Every velocity of one axis of one sign (no group of the other)."""
    check(wl._case(2, [20, 18], 2.0, 8, ([0.1, -4.0], [6.0, 4.0]), 0.2, 2.0, {"kind": "none"}))


def test_slabs_of_rows():
    """Tables of more than 256 MB: the grid is swept in slabs of rows."""
    check(wl._case(2, [2000, 600], 8.0, 8, 4.0, 0.2, 0.3, wl.circle(0.5)), steps=1,
          threads=min(16, os.cpu_count() or 1))
