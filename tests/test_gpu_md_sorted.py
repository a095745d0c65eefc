"""MD segments with the particles sorted by cell (Nmax up to 512) against the
cell list (Nmax 513): the same walkers end in the same positions, kinetic and
potential energies, bit for bit -- at particle counts around the warps and the
CTA, in rectangular, sheared, fully periodic and one-cell-wide boxes."""
import numpy as np
import pytest

import workloads as W
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu

SORTED, LISTED = 512, 513


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def fcc111(nmax):
    p = W.fcc111_paper_scale(L=2, M=4, nmax=nmax)
    return p, *W.lattice_walkers(p, np.array([0, 1, 31, 33, 127, 128, 129, 511]), seed=1)


def fcc100(nmax):
    p = W.fcc100_small(L=2, M=2, nmax=nmax)
    return p, *W.lattice_walkers(p, np.array([0, 5, 32, 100]), seed=2)


def minimal_periods(nmax):
    xyz, lx, ly, ztop = W.fcc100_slab(4, 4, 2, 1.25)
    p = W.fcc100_small(L=2, M=2, nmax=nmax).replace(
        Lx=5.0, Ly=5.0, surf_xyz=xyz, surf_type=np.ones(len(xyz), np.int32), z_lo=ztop, z_hi=ztop + 9.0)
    return p, *W.lattice_walkers(p, np.array([1, 8, 31, 60]), seed=3)


def hexagonal(nmax):
    p = W.lj_a18_hex_slab(L=2, M=2, nmax=nmax)
    return p, *W.lj_a18_initial(p, np.array([0, 12, 33, 50]), seed=4)


def cluster(nmax):
    p = W.cluster_in_gas(L=2, M=2, nmax_b=nmax - 4)
    return p, *W.cluster_initial(p, np.array([0, 1, 124, 500]), seed=5)


@pytest.mark.parametrize("system", [fcc111, fcc100, minimal_periods, hexagonal, cluster])
def test_sorted_and_listed_segments_are_the_same(system):
    got = []
    for nmax in (SORTED, LISTED):
        p, pos, n = system(nmax)
        g = Regc(p)
        g.set_walkers(pos, n)
        kin = [g.md(4, 0.002, 0.1) for _ in range(2)]
        x, m, e, _ = g.get_walkers()
        assert np.array_equal(m, n)
        got.append((kin, e, [x[w, :k] for w, k in enumerate(m)]))
    (ka, ea, xa), (kb, eb, xb) = got
    assert all(np.array_equal(u, v) for u, v in zip(ka, kb))
    assert np.array_equal(ea, eb)
    assert all(np.array_equal(u, v) for u, v in zip(xa, xb))
    assert all(np.isfinite(u).all() for u in xa)
