"""The enumeration over all particles against the cell list (launch.h:
direct_limit): the same walkers and seed in a handle whose Nmax is at the limit
and in one with Nmax 161 (always cells) make the same moves, bit for bit, while
N stays below the smaller Nmax (Nmax enters a move only at N = Nmax).  Over the
forms the rule accepts: rectangular, sheared and fully periodic cells, a
cluster, two species, periods of exactly 2 rc (one cell along an axis), few and
many walkers per SM, every number of warps per walker."""
import numpy as np
import pytest

import workloads as W
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu

CELLS = 161
LOW_MU = np.array([-9.0, -8.0, -7.0, -6.0])   # the walkers empty rather than fill up to Nmax


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def _start(p, n, seed):
    """Walkers of p with at most its region's lattice sites."""
    return W.lattice_walkers(p, np.minimum(n, int(0.9 * W.lattice_sites(p))), seed=seed)


def fcc111(nmax):
    p = W.fcc111_paper_scale(L=2, M=4, nmax=nmax).replace(mu=LOW_MU - 8.0)
    return p, *_start(p, np.array([0, 1, 5, 16, 31, 32, 33, 34]), 1), None


def fcc100(nmax):
    p = W.fcc100_small(L=2, M=4, nmax=nmax)
    return p, *_start(p, np.array([0, 1, 5, 16, 31, 32, 33, 40]), 2), None


def minimal_periods(nmax):
    """Periods of exactly 2 rc along x and y: one cell, every image at a tie."""
    xyz, lx, ly, ztop = W.fcc100_slab(4, 4, 2, 1.25)
    p = W.fcc100_small(L=2, M=4, nmax=nmax).replace(
        Lx=5.0, Ly=5.0, rc=2.5, surf_xyz=xyz, surf_type=np.ones(len(xyz), np.int32), z_lo=ztop, z_hi=ztop + 9.0)
    return p, *_start(p, np.array([0, 1, 8, 16, 24, 31, 32, 33]), 3), None


def hexagonal(nmax):
    p = W.lj_a18_hex_slab(L=2, M=4, nmax=nmax)
    pos, n = W.lj_a18_initial(p, np.array([0, 1, 12, 18, 24, 33, 40, 50]), seed=4)
    return p, pos, n, None


def cluster(nmax):
    p = W.cluster_in_gas(L=2, M=4, nmax_b=nmax - 4).replace(mu=LOW_MU - 4.0)
    pos, n = W.cluster_initial(p, np.array([0, 1, 5, 16, 27, 28, 29, 30]), seed=5)
    return p, pos, n, None


def cluster_many(nmax):
    p = W.cluster_in_gas(L=32, M=64, nmax_b=nmax - 4).replace(mu=np.linspace(-14.0, -10.0, 64))
    pos, n = W.cluster_initial(p, np.random.default_rng(0).integers(0, 101, p.S), seed=7)
    return p, pos, n, None


def two_gas(nmax):
    p = W.two_gas_small(L=2, M=2, K=2, nmax=nmax)
    pos, n = _start(p, np.array([0, 1, 5, 16, 31, 32, 33, 40]), 6)
    return p, pos, n, (n // 2).astype(np.int32)


# the largest Nmax of the direct enumeration: 160, or 96 ncell / (ncell - 27)
# with few walkers per SM and more than 27 cells (168 and 125 here)
@pytest.mark.parametrize("system,limit", [(fcc111, 114), (fcc100, 160), (minimal_periods, 160), (hexagonal, 160),
                                          (cluster, 122), (cluster_many, 160), (two_gas, 160)])
@pytest.mark.parametrize("warps", [1, 2, 4])
def test_direct_and_cells_make_the_same_moves(system, limit, warps, monkeypatch):
    monkeypatch.setenv("REGC_WARPS_PER_WALKER", str(warps))
    got = []
    for nmax in (limit, CELLS):
        p, pos, n, nb = system(nmax)
        g = Regc(p)
        g.set_walkers(pos, n, nb=nb)
        for _ in range(4):
            g.sweep(10)
            g.exchange()
        # N cannot have reached the limit between two observations (20 moves apart)
        hN = g.histograms()["hN"].sum(axis=0)
        assert np.nonzero(hN)[0].max() + p.n_cluster + p.moves_per_sweep < limit
        x, m, e, sow = g.get_walkers()
        mv, ex, pr = g.counters()
        got.append((m, e, sow, mv, ex, pr[0], [x[w, :k] for w, k in enumerate(m)], g.check_energy()))
    a, b = got
    for u, v in zip(a[:6], b[:6]):
        assert np.array_equal(u, v)
    assert all(np.array_equal(u, v) for u, v in zip(a[6], b[6]))
    assert a[7] == 0.0 and b[7] == 0.0
    assert a[3].sum() > 0


def test_direct_capacity_is_refused():
    """A cell beyond the cell list's capacity (43 here) is refused by the direct
    enumeration too."""
    p = W.fcc111_paper_scale(L=1, M=1, nmax=61).replace(eps=np.zeros((4, 4)))
    g = np.arange(4) * 0.6 + 0.15
    sites = [(x, y, p.z_lo + z) for z in np.arange(4) * 0.55 + 1.0 for y in g for x in g]
    pos = W.f32(sites[:61])[None]
    for k, refused in ((43, False), (44, True)):
        h = Regc(p.replace(p_disp=1.0, max_disp=0.0))
        h.set_walkers(pos, np.array([k], np.int32))
        h.sweep(1)
        if refused:
            with pytest.raises(Exception):
                h.get_walkers()
        else:
            assert h.get_walkers()[1][0] == k
