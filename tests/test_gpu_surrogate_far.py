"""The surrogate's features with cut-offs beyond the reach of its Gaussians (the
last centre is 2.5, their width 0.113): a neighbour far away adds nothing, and
delayed acceptance screens with finite energies."""
import numpy as np
import pytest

import workloads as W
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def empty_box(rc, nmax=8, **kw):
    return W.fcc100_small(L=1, M=1, nmax=nmax).replace(
        rc=rc, Lx=40.0, Ly=40.0, z_lo=0.0, z_hi=40.0, surf_xyz=np.zeros((0, 3)), surf_type=np.zeros(0, np.int32), **kw)


@pytest.mark.parametrize("rc", [2.5, 9.9, 11.0, 11.5, 14.0, 19.9])
def test_far_neighbours_add_nothing(rc):
    """exp(-eta (r - 2.5)^2) is below 2^-149 from r = 4.13 on."""
    g = Regc(empty_box(rc))
    g.surrogate_init(1)
    pos = np.zeros((1, 8, 3))
    pos[0, 0] = (20.0, 20.0, 20.0)
    g.set_walkers(pos, np.array([1], np.int32))
    r = np.concatenate([np.arange(4.2, 19.9, 0.05), [9.9999, 10.0, 10.0001, 11.36, 11.37, 11.38]])
    e, F = g.surrogate_eval(0, np.stack([20.0 - r, 0 * r + 20.0, 0 * r + 20.0], 1))
    lone, _ = g.surrogate_eval(0, [[0.0, 0.0, 0.0]])
    assert np.array_equal(F, np.zeros_like(F))
    assert np.array_equal(e, np.full_like(e, lone[0]))


def test_screening_with_a_long_cutoff():
    """Two particles 12 apart with rc = 14: the screen sees the energy of a lone
    particle at both ends of a move, so every displacement passes it."""
    p = empty_box(14.0, p_disp=1.0, max_disp=0.05)
    g = Regc(p)
    g.surrogate_init(1)
    g.set_mode(True)
    pos = np.zeros((1, 8, 3))
    pos[0, 0], pos[0, 1] = (14.0, 20.0, 20.0), (26.0, 20.0, 20.0)
    g.set_walkers(pos, np.array([2], np.int32))
    g.sweep(10)
    _, _, pairs = g.counters()
    assert pairs[4] == pairs[5] == 10 * p.moves_per_sweep
    assert g.check_energy() == 0.0
