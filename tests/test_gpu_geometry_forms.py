"""The walk compiled for a geometry (launch.h: sweep_geo) against the general
form, which traced sweeps run: the same walkers and seed make the same moves,
bit for bit, on slabs, sheared slabs and periodic boxes, with one species, two
and a cluster, through the cell list and the direct enumeration, with every
number of warps per walker."""
import numpy as np
import pytest

import workloads as W
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def periodic(p, edge=12.5):
    """p in a cube without its surface."""
    return p.replace(Lx=edge, Ly=edge, Lz=edge, periodic_z=1, z_lo=0.0, z_hi=edge, surf_xyz=np.zeros((0, 3)),
                     surf_type=np.zeros(0, np.int32))


def sheared(p):
    return p.replace(shear=0.5, Lx=p.Lx * 1.25)


def system(name, nmax):
    n = np.array([0, 5, 20, 40])
    if name == "cluster":
        p = W.cluster_in_gas(L=2, M=2, nmax_b=nmax - 4)
        return p, *W.cluster_initial(p, n, seed=5), None
    if name == "hexagonal":
        p = W.lj_a18_hex_slab(L=2, M=2, nmax=nmax)
        return p, *W.lj_a18_initial(p, n, seed=4), None
    p = W.two_gas_small(L=2, M=2, K=1, nmax=nmax) if "two" in name else W.fcc111_paper_scale(L=2, M=2, nmax=nmax)
    if "periodic" in name:
        p = periodic(p)
    if "sheared" in name:
        p = sheared(p)
    pos, n = W.lattice_walkers(p, np.minimum(n, int(0.9 * W.lattice_sites(p))), seed=1)
    return p, pos, n, (n // 2).astype(np.int32) if "two" in name else None


@pytest.mark.parametrize("name", ["slab", "sheared", "periodic", "hexagonal", "cluster", "two", "two sheared",
                                  "two periodic"])
@pytest.mark.parametrize("nmax", [50, 200])   # direct, cells
@pytest.mark.parametrize("warps", [1, 2, 4])
def test_compiled_geometry_makes_the_general_forms_moves(name, nmax, warps, monkeypatch):
    monkeypatch.setenv("REGC_WARPS_PER_WALKER", str(warps))
    p, pos, n, nb = system(name, nmax)
    got = []
    for traced in (False, True):
        g = Regc(p)
        g.set_walkers(pos, n, nb=nb)
        for _ in range(3):
            g.sweep_traced(20) if traced else g.sweep(20)
            g.exchange()
        x, m, e, sow = g.get_walkers()
        mv, ex, pr = g.counters()
        got.append((m, e, sow, mv, ex, pr, np.concatenate([x[w, :k] for w, k in enumerate(m)])))
        assert g.check_energy() == 0.0
        g.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert got[0][3].sum() > 0
