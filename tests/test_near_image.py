"""The nearest-image difference of the direct enumeration, in binary32 on the
CPU, against the images of the cell stencil (query or partner shifted by the
period, one rounding): in-range differences are the same bit for bit, at ties
of half a period and for periods of exactly 2 rc too."""
import numpy as np
import pytest

F = np.float32


def near_diff(q, p, L):
    hL = F(0.5) * L
    e = (q - p).astype(F)
    qs = np.where(e >= hL, (q - L).astype(F), q)
    ps = np.where(e <= -hL, (p - L).astype(F), p)
    return (qs - ps).astype(F)


def images(q, p, L):
    """The stencil's three images: plain, query shifted, partner shifted."""
    return (q - p).astype(F), ((q - L).astype(F) - p).astype(F), (q - (p - L).astype(F)).astype(F)


@pytest.mark.parametrize("L", [5.0, 5.0000005, 6.25, 11.489, 15.0, 18.75])
def test_in_range_differences_equal_the_stencils(L):
    L, rc = F(L), F(2.5)
    rng = np.random.default_rng(7)
    q = (rng.random(400000) * L).astype(F)
    p = (rng.random(400000) * L).astype(F)
    # half of them at the tie of half a period, to the last bits
    k = len(q) // 2
    p[:k] = ((q[:k].astype(np.float64) + 0.5 * float(L) + rng.integers(-3, 4, k) * 2.0 ** -23) % float(L)).astype(F)
    q, p = np.minimum(q, np.nextafter(L, F(0))), np.minimum(p, np.nextafter(L, F(0)))
    d = near_diff(q, p, L)
    im = images(q, p, L)
    inside = [np.abs(x) < rc for x in im]
    # at most one image is within rc, and it is the one taken
    assert not np.any(sum(i.astype(int) for i in inside) > 1)
    for x, i in zip(im, inside):
        assert np.array_equal(d[i], x[i])
    assert np.array_equal(np.abs(d) < rc, inside[0] | inside[1] | inside[2])
