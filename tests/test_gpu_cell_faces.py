"""The walk where its cell geometry is hardest: particles at the faces of cells to
the last bits and around rc from each other, walls far from the origin, one, two
and more cells along an axis, rectangular, sheared and fully periodic.  The cell
list (whose stencil leaves out cells out of reach), its general form (traced
sweeps, the same rule) and the enumeration of all particles (nearest images, no
cells) end in the same state bit for bit, and the running energies equal the
from-scratch ones, which know no such rule."""
import numpy as np
import pytest

import workloads as W
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu

DIRECT, CELLS = 90, 200   # Nmax below and above the enumeration of all particles


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def at_faces(rng, n, lo, L, k):
    """n coordinates in [lo, lo + L), half of them at faces of the k cells to the last bits."""
    x = lo + rng.random(n) * L
    h = rng.random(n) < 0.5
    x[h] = (lo + L / k * rng.integers(0, k + 1, n) + rng.integers(-3, 4, n) * np.spacing(np.float32(abs(lo) + L)))[h]
    return np.clip(x.astype(np.float32), np.float32(lo), np.nextafter(np.float32(lo + L), np.float32(lo)))


def walkers(p, k, count, rng):
    """Particles at faces, every other one around rc from an earlier one, 0.9 apart."""
    L, lo = np.array([p.Lx, p.Ly, p.z_hi - p.z_lo]), np.array([0.0, 0.0, p.z_lo])
    per = np.array([True, True, bool(p.periodic_z)])
    out = []
    for i in range(60 * count):
        q = np.array([at_faces(rng, 1, lo[a], L[a], k[a])[0] for a in range(3)], np.float64)
        if out and i % 2:
            d = rng.normal(size=3)
            d *= p.rc * rng.choice([0.9999, 1.0, 1.0001]) / np.linalg.norm(d)
            d[0] -= p.shear * d[1]
            q = out[rng.integers(len(out))] + d
            q = np.where(per, lo + np.mod(q - lo, L), q)
        q = q.astype(np.float32).astype(np.float64)
        if np.any(q < lo.astype(np.float32)) or np.any(q >= (lo + L).astype(np.float32)):
            continue
        d = np.array(out).reshape(-1, 3) - q
        d -= np.where(per, L * np.round(d / L), 0.0)
        d[:, 0] += p.shear * d[:, 1]
        if np.all(np.sum(d * d, 1) > 0.81):
            out.append(q)
        if len(out) == count:
            break
    return np.array(out)


# Lx, Ly, z_lo, height, rc, shear, periodic z
@pytest.mark.parametrize("Lx,Ly,z0,hz,rc,shear,per", [
    (15.0, 17.3205, 0.9, 14.0, 2.5, 0.0, 0),
    (5.0, 5.0, 0.9, 9.0, 2.5, 0.0, 0),
    (7.51, 9.99, -3.0, 2.0, 2.5, 0.0, 0),
    (40.0, 31.0, 1000.0, 30.0, 2.9, 0.0, 0),
    (12.5, 12.5, 0.0, 12.5, 2.5, 0.0, 1),
    (5.0, 7.6, 0.0, 5.1, 2.5, 0.0, 1),
    (8.0, 6.9282, 1.1, 8.0, 2.5, 0.5, 0),
    (9.0, 8.0, 0.0, 6.0, 2.0, -0.5, 1),
])
@pytest.mark.parametrize("warps", [1, 4])
def test_cells_and_all_particles_make_the_same_moves(Lx, Ly, z0, hz, rc, shear, per, warps, monkeypatch):
    monkeypatch.setenv("REGC_WARPS_PER_WALKER", str(warps))
    rng = np.random.default_rng(3)
    gx, gy = np.meshgrid((np.arange(6) + 0.5) * Lx / 6, (np.arange(6) + 0.5) * Ly / 6)
    atoms = np.zeros((0, 3)) if per else np.stack([gx.ravel(), gy.ravel(), np.full(36, z0 - 0.9)], 1)
    p = W.fcc111_paper_scale(L=2, M=2, nmax=CELLS).replace(
        Lx=Lx, Ly=Ly, Lz=hz if per else 0.0, periodic_z=per, z_lo=z0, z_hi=z0 + hz, rc=rc, shear=shear,
        surf_xyz=atoms, surf_type=np.ones(len(atoms), np.int32), mu=np.array([-16.0, -14.0]), p_disp=0.9, max_disp=0.3)
    if per:
        p = p.replace(z_hi=p.Lz)
    su = np.sqrt(1.0 + shear * shear)
    k = [max(1, int(np.floor(n / (r * 1.00001)))) for n, r in zip((Lx, Ly, hz), (rc * su, rc, rc))]
    pos, n = np.zeros((4, CELLS, 3)), np.zeros(4, np.int32)
    for w in range(4):
        q = walkers(p, k, 15 * (w + 1), rng)
        pos[w, :len(q)], n[w] = q, len(q)
    assert n.max() > 20
    got = []
    for nmax, traced in ((DIRECT, False), (CELLS, False), (CELLS, True)):
        g = Regc(p.replace(nmax=nmax))
        g.set_walkers(pos[:, :nmax], n)
        for _ in range(3):
            g.sweep_traced(10) if traced else g.sweep(10)
            g.exchange()
            assert g.check_energy() == 0.0
        x, m, e, sow = g.get_walkers()
        mv, _, pr = g.counters()
        assert m.max() < DIRECT - p.moves_per_sweep
        got.append((m, e, sow, mv, pr[0], np.concatenate([x[w, :c] for w, c in enumerate(m)])))
        g.close()
    for a, b, c in zip(*got):
        assert np.array_equal(a, b) and np.array_equal(b, c)
    assert got[0][3][:, :, 1].sum() > 100
