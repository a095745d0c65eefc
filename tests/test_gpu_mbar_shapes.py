"""The sparse kernel matrix at the edges of its tiles: numbers of states around
a word of 32, around the 448 whose weights travel with the launch, and numbers
of bins around a warp's 32 and a chunk; the device solution is a fixed point of
the oracle's own map, with the same D_b, and the query over runs agrees with
the oracle's."""
import math

import numpy as np
import pytest

from oracle import mbar as OM
from paper_1908_11118_gb300 import build as B
from paper_1908_11118_gb300 import mbar_last_info, mbar_query, mbar_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def model_bins(S, bins, seed):
    """S states on a line through the (kT, mu) plane over exactly `bins` bins of a
    model density of states (every state overlaps its neighbours)."""
    rng = np.random.default_rng(seed)
    kT = np.linspace(0.9, 1.4, S)
    mu = np.linspace(-4.0, -3.0, S)
    N = np.sort(rng.integers(0, 25, bins))
    E = np.round((-2.0 * N + rng.normal(size=bins) * (0.5 + 0.3 * np.sqrt(N))) * 50.0) / 50.0
    lnw = (-(E[None] - mu[:, None] * N[None]) / kT[:, None] + N[None] * (1.5 * np.log(kT)[:, None] + math.log(100.0))
           - np.array([math.lgamma(k + 1) for k in N])[None])
    w = np.exp(lnw - lnw.max(axis=1, keepdims=True))
    omega = rng.integers(500, 3000, S).astype(float)
    H = (omega[:, None] * w / w.sum(axis=1, keepdims=True)).sum(axis=0) + 1e-6
    return kT, mu, omega * H.sum() / omega.sum(), N, E, H


@pytest.mark.parametrize("S,bins", [(1, 1), (1, 40), (2, 31), (31, 32), (32, 33), (33, 64), (64, 1000), (447, 300),
                                    (448, 301), (449, 300), (1025, 97), (3, 20000), (40, 70001)])
def test_matrix_shapes(S, bins):
    kT, mu, omega, N, E, H = model_bins(S, bins, seed=S + bins)
    f, D, _ = mbar_solve(kT, mu, 1.0, omega, N, E, H, tol=1e-11)
    info = mbar_last_info()
    assert info["path"] == 1 and info["lse_maps"] == 0
    assert 0 < info["nnz"] <= S * bins
    # one FP64 map of the oracle from f stays there (the convergence asked for,
    # 1e-11, and the rounding of sums of up to 7e4 terms of size e^+-100)
    f1, D1, _, _ = OM.solve(kT, mu, 1.0, omega, N, E, H, max_iter=1, f0=f)
    np.testing.assert_allclose(f, f1, atol=1e-9)
    np.testing.assert_allclose(D, D1, atol=1e-9)
    kq, mq = np.array([0.95, 1.2]), np.array([-3.8, -3.1])
    n_o, p_o, fq_o = OM.query(kq, mq, 1.0, N, E, H, D, 30)
    n_g, p_g, fq_g = mbar_query(kq, mq, 1.0, N, E, H, D, 30)
    np.testing.assert_allclose(n_g, n_o, rtol=1e-9, atol=1e-12)
    np.testing.assert_allclose(p_g, p_o, atol=1e-10)
    np.testing.assert_allclose(fq_g, fq_o, atol=1e-9)
