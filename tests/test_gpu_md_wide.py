"""MD segments in boxes of many cells, whose counts are scanned a run of cells per
lane (more than 256 cells), against the cell list of Nmax 513: the same walkers end
in the same positions and energies, bit for bit, at cell counts around the rule's
line and around multiples of 32, nearly empty and full, with a cluster too."""
import numpy as np
import pytest

import workloads as W
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("cells", [(4, 8, 8), (1, 1, 257), (5, 8, 7), (2, 16, 9), (11, 3, 9), (12, 12, 12)])
@pytest.mark.parametrize("cluster", [False, True])
def test_many_cells(cells, cluster):
    rng = np.random.default_rng(sum(cells))
    edge = np.array([max(5.01, 2.51 * c) for c in cells])
    cells = [int(e / (2.5 * 1.00001)) for e in edge]
    counts = np.array([4, 40, 129, 500])
    got = []
    for nmax in (512, 513):
        p = (W.cluster_in_gas(L=2, M=2, nmax_b=nmax - 4) if cluster else W.fcc111_paper_scale(L=2, M=2, nmax=nmax))
        p = p.replace(Lx=edge[0], Ly=edge[1], Lz=edge[2], periodic_z=1, z_lo=0.0, z_hi=edge[2], rc=2.5,
                      surf_xyz=np.zeros((0, 3)), surf_type=np.zeros(0, np.int32))
        p = p.replace(z_hi=p.Lz)
        if nmax == 512:
            k = np.maximum(1, (edge / 1.25).astype(int))
            n = np.minimum(counts, int(0.9 * np.prod(k)))
            pos = np.zeros((4, 512, 3))
            for w in range(4):
                q = rng.choice(int(np.prod(k)), n[w], replace=False)
                pos[w, :n[w]] = (np.stack([q % k[0], q // k[0] % k[1], q // (k[0] * k[1])], 1) + 0.5) * (edge / k)
        x0 = np.zeros((4, nmax, 3))
        x0[:, :512] = pos
        g = Regc(p)
        g.set_walkers(x0, n.astype(np.int32))
        kin = [g.md(3, 0.002, 0.1) for _ in range(2)]
        x, m, e, _ = g.get_walkers()
        got.append((kin, e, [x[w, :c] for w, c in enumerate(m)]))
        g.close()
    (ka, ea, xa), (kb, eb, xb) = got
    assert all(np.array_equal(u, v) for u, v in zip(ka, kb))
    assert np.array_equal(ea, eb)
    assert all(np.array_equal(u, v) for u, v in zip(xa, xb))
    assert all(np.isfinite(u).all() for u in xa)
