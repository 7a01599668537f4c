"""Waiting for a plan's work: a thread that waits long gives up its core, with and without a limit."""
import time

import numpy as np
import pytest

import paper_0812_3669_gb300 as moff

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    moff.build()
    yield


@pytest.mark.parametrize("timeout_ms", [-1, 60000])
def test_a_long_wait_leaves_the_core(timeout_ms):
    N, A, P, C, T = 512, 64, 2, 16, 128
    rng = np.random.default_rng(3)
    pos, taps = rng.uniform(0, N, size=(A, 2)), np.ones((A, P, 3, 3), np.complex64)
    codes = torch.randint(0, 256, (T, C, A, P), dtype=torch.uint8, device="cuda")
    with moff.Plan(pos, taps, N, C, P) as pl:
        pl.submit(codes)
        pl.sync()
        n, wall = 32, 0.0
        while wall < 0.2:                     # blocks enqueued ahead until the wait is long
            n *= 2
            for _ in range(n):
                pl.submit(codes)
            t0, c0 = time.perf_counter(), time.thread_time()
            pl.sync(timeout_ms)
            wall, cpu = time.perf_counter() - t0, time.thread_time() - c0
            assert n < 1 << 16
    assert cpu < 0.5 * wall, (cpu, wall)
