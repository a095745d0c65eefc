"""The sparse kernel matrix at the limits of its indices, of the memory it may
take and of its waits."""
import ctypes
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from oracle import mbar as OM
from paper_1908_11118_gb300 import build as B
from paper_1908_11118_gb300 import mbar_last_info, mbar_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def close_states(S, bins, seed):
    """S states so close in (kT, mu) that every bin keeps the terms of all of them."""
    rng = np.random.default_rng(seed)
    kT, mu = np.linspace(1.0, 1.05, S), np.linspace(-3.5, -3.4, S)
    N = np.sort(rng.integers(0, 25, bins))
    E = -2.0 * N + rng.normal(size=bins) * (0.5 + 0.3 * np.sqrt(N))
    H = rng.uniform(1.0, 50.0, bins)
    return kT, mu, np.full(S, H.sum() / S), N, E, H


@pytest.mark.parametrize("S", [65536, 65537, 65600])
def test_rows_of_more_than_65535_states(S):
    """The number of a row's entries before a word of 32 states passes 65535."""
    kT, mu, omega, N, E, H = close_states(S, 40, seed=S)
    f, D, _ = mbar_solve(kT, mu, 1.0, omega, N, E, H, tol=1e-11)
    info = mbar_last_info()
    assert info["path"] == 1 and info["lse_maps"] == 0 and info["nnz"] == S * len(N)
    # one FP64 map of the oracle from f stays there (the convergence asked for,
    # 1e-11, and the rounding of sums of up to 7e4 terms of size e^+-100)
    f1, D1, _, _ = OM.solve(kT, mu, 1.0, omega, N, E, H, max_iter=1, f0=f)
    np.testing.assert_allclose(f, f1, atol=1e-9)
    np.testing.assert_allclose(D, D1, atol=1e-9)


class Pool:
    """The most that the device's default memory pool held at once since reset()."""
    USED_MEM_HIGH = 8

    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        dev, self.pool = ctypes.c_int(), ctypes.c_void_p()
        assert self.cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), dev) == 0

    def reset(self):
        assert self.cu.cuMemPoolSetAttribute(self.pool, self.USED_MEM_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0

    def high(self):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, self.USED_MEM_HIGH, ctypes.byref(v)) == 0
        return v.value


def test_masks_count_against_half_the_free_memory():
    """1.2e6 bins of 4096 states take 0.9 GB or more of masks: with 1.6 GB free the
    solve does without the matrix and never holds half of what is free."""
    torch = pytest.importorskip("torch")
    left = 1_600_000_000
    torch.cuda.init()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        kT, mu, omega, N, E, H = close_states(4096, 1_200_000, seed=1)
        pool = Pool()
        torch.cuda.synchronize()
        pool.reset()
        mbar_solve(kT, mu, 1.0, omega, N, E, H, max_iter=1)
        assert pool.high() < left // 2
        assert mbar_last_info()["path"] == 0
    finally:
        del hold
        torch.cuda.empty_cache()


BLOCKING = """
import ctypes, time
import numpy as np
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0     # blocking waits
from paper_1908_11118_gb300 import mbar_last_info, mbar_solve
rng = np.random.default_rng(0)
S, B = 64, 1000000
N = np.sort(rng.integers(0, 25, B))
E, H = -2.0 * N + rng.normal(size=B), rng.uniform(1.0, 5.0, B)
a = (np.linspace(0.9, 1.4, S), np.linspace(-4.0, -3.0, S), 1.0, np.full(S, H.sum() / S), N, E, H)
mbar_solve(*a, max_iter=3)
wall, cpu = time.perf_counter(), time.thread_time()
mbar_solve(*a, tol=1e-300, max_iter=400)
wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
assert mbar_last_info()["sparse_maps"] == 400
print(wall, cpu)
"""


def test_the_waits_follow_the_scheduling_flags():
    """With blocking waits set for the device, a solve of 400 maps of 0.3 ms leaves
    its core to others: less than half of the wall time is its own."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", BLOCKING], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    wall, cpu = (float(v) for v in r.stdout.split())
    assert cpu < 0.5 * wall


def test_a_solve_does_not_wait_for_other_streams():
    """After a first solve, solves (of more states, and of a thread of their own) end
    while another stream still runs a kernel of some 0.2 s."""
    torch = pytest.importorskip("torch")
    small, large = close_states(64, 2000, seed=2), close_states(1024, 2000, seed=3)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()

    def solve(a):
        mbar_solve(*a[:2], 1.0, *a[2:], tol=1e-300, max_iter=20, stream=mine)

    solve(small)
    thread = threading.Thread(target=lambda: (solve(small), solve(large)))
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(400_000_000)
        end = torch.cuda.Event()
        end.record(other)
    solve(small)
    solve(large)
    thread.start()
    thread.join()
    running = not end.query()
    torch.cuda.synchronize()
    assert running


def test_threads_share_the_page_locked_memory():
    """Solves of different sizes in eight threads at once equal the same solves alone."""
    problems = [close_states(S, 500 + S, seed=S) for S in (1, 30, 64, 300, 449, 700, 1024, 5000)]

    def solve(a):
        return mbar_solve(*a[:2], 1.0, *a[2:], tol=1e-11)

    alone = [solve(a) for a in problems]
    got = [[None] * len(problems) for _ in range(3)]

    def work(k):
        for turn in got:
            turn[k] = solve(problems[k])

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(problems))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for turn in got:
        for (f, D, it), (g, E, jt) in zip(alone, turn):
            assert np.array_equal(f, g) and np.array_equal(D, E) and it == jt


RESET = """
import ctypes
import numpy as np
from paper_1908_11118_gb300 import mbar_solve
rng = np.random.default_rng(0)
S, B = 64, 2000
N = np.sort(rng.integers(0, 25, B))
E, H = -2.0 * N + rng.normal(size=B), rng.uniform(1.0, 5.0, B)
a = (np.linspace(0.9, 1.4, S), np.linspace(-4.0, -3.0, S), 1.0, np.full(S, H.sum() / S), N, E, H)
first = mbar_solve(*a)
assert ctypes.CDLL("libcuda.so.1").cuDevicePrimaryCtxReset_v2(0) == 0     # this process's own context
again = mbar_solve(*a)
assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])
"""


def test_a_solve_after_the_context_was_reset():
    """The page-locked memory kept from a solve goes with its context."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
