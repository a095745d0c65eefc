"""The rule that leaves a cell of the stencil out of the enumeration (walker.cuh:
stencil_list), in binary32 on the CPU against all images of the stencil: a cell
that holds a partner within rc of a query is never left out, for rectangular,
sheared and fully periodic cells, one, two and more cells along an axis, walls
far from the origin, and coordinates at the faces of cells."""
import numpy as np
import pytest

F = np.float32


def at_faces(rng, n, lo, L, k):
    """n coordinates in [lo, lo + L): half of them at faces of the k cells, to the last bits."""
    x = lo + rng.random(n) * L
    h = n // 2
    x[:h] = lo + L / k * rng.integers(0, k, h) + rng.integers(-3, 4, h) * np.spacing(F(abs(lo) + L))
    return np.clip(x.astype(F), F(lo), np.nextafter(F(lo + L), F(lo)))


# Lx, Ly, z_lo, height, rc, shear, periodic z
@pytest.mark.parametrize("Lx,Ly,z0,hz,rc,shear,per", [
    (15.0, 17.3205, 0.9, 14.0, 2.5, 0.0, False),
    (5.0, 5.0, 0.9, 9.0, 2.5, 0.0, False),
    (7.51, 9.99, -3.0, 2.0, 2.5, 0.0, False),
    (40.0, 31.0, 1000.0, 30.0, 2.9, 0.0, False),
    (12.5, 12.5, 0.0, 12.5, 2.5, 0.0, True),
    (5.0, 7.6, 0.0, 5.1, 2.5, 0.0, True),
    (8.0, 6.9282, 1.1, 8.0, 2.5, 0.5, False),
    (9.0, 8.0, 0.0, 6.0, 2.0, -0.5, True),
])
def test_no_cell_with_a_partner_in_range_is_left_out(Lx, Ly, z0, hz, rc, shear, per):
    rng = np.random.default_rng(11)
    su = np.sqrt(1 + shear * shear)
    L = np.array([Lx, Ly, hz])
    lo = np.array([0.0, 0.0, 0.0 if per else z0])
    k = np.array([max(1, int(np.floor(n / (r * 1.00001)))) for n, r in zip(L, (rc * su, rc, rc))])
    ic = (k / L).astype(F)
    w = (F(1) / ic).astype(F)
    zs = F(hz) if per else F(abs(z0)) + F(abs(z0 + hz))
    reach = F(rc) * F(1.001) + F(2e-6) * (F(Lx) + F(Ly) + zs)
    n = 60000
    q = np.stack([at_faces(rng, n, lo[a], L[a], k[a]) for a in range(3)], 1)
    # partners around rc of their query, then into the cell (or dropped beyond the walls)
    d = rng.normal(size=(n, 3))
    d *= (rc * rng.choice([0.3, 0.9, 0.9999, 1.0], n) / np.linalg.norm(d, axis=1))[:, None]
    d[:, 0] -= shear * d[:, 1]
    p = q.astype(np.float64) + d
    for a in range(2 + per):
        p[:, a] = np.mod(p[:, a], L[a])
    p = p.astype(F)
    keep = np.all((p >= lo.astype(F)) & (p < (lo + L).astype(F)), axis=1)
    q, p = q[keep], p[keep]

    def cell(x):
        rel = x - (np.array([0, 0, 0 if per else z0])).astype(F)
        return np.clip((rel * ic).astype(np.int64), 0, k - 1)

    cq, cp = cell(q), cell(p)
    corner = (cq.astype(F) * w + lo.astype(F)).astype(F)
    f = (corner - q).astype(F)
    found = np.zeros(len(q), bool)
    for o in np.ndindex(3, 3, 3):
        off = np.array(o) - 1
        at = cq + off
        wrap = np.where(at < 0, -1, np.where(at >= k, 1, 0))
        listed = np.all(cq + off - wrap * k == cp, axis=1) & (per | (wrap[:, 2] == 0))
        e = q.astype(np.float64) - (p.astype(np.float64) + wrap * L)
        e[:, 0] += shear * e[:, 1]
        in_range = listed & (np.sum(e * e, 1) < rc * rc * (1 + 1e-6))
        a = np.abs(off).astype(F)
        b = np.where(off > 0, w, F(0)).astype(F)
        if shear:
            a[0] = b[0] = F(0)
        gap = (a * f + b).astype(F)
        taken = np.sum(gap * gap, 1, dtype=F) < reach * reach
        assert np.all(taken[in_range])
        found |= in_range
    assert found.sum() > len(q) // 2
