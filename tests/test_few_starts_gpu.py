"""Starts where few can start at once, on the GPU against the oracle: one to four
slots, KV for one to four of the longest requests, queues of one to four, and a
queue whose only request shares its length with others that are not there yet."""
import numpy as np
import pytest

from conftest import cuda_available
from test_parity_gpu import INF, O, S, run_both  # noqa: F401  (fixtures)

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]

RUNS = ["ljf", "sjf", "isjl", "isjl", "isjl", "isjl_beta", "fcfs"], [0, 0, 0, 30, INF, 30, 0]


@pytest.mark.parametrize("B", [1, 2, 3, 4, 9, 40])
def test_kv_around_a_few_of_the_longest(S, O, B):  # noqa: F811
    rng = np.random.default_rng(B)
    n = 90                                              # more than a thread per task takes
    o = np.stack([rng.integers(1, 200, n), rng.choice([100, 60, 20], n), np.full(n, 100),
                  rng.integers(90, 101, n)]).astype(np.int32)
    o[:, 0] = 100
    o = np.minimum(o, 100)
    p = np.zeros_like(o)
    a = np.zeros_like(o)
    a[1] = np.sort(rng.integers(0, 100 * n // B, n))
    for kv in (100, 199, 200, 299, 300, 301, 400, INF):
        run_both(S, O, a, p, o, B, *RUNS, kv)
    e = rng.integers(0, 40, o.shape).astype(np.int32)
    run_both(S, O, a, p, o, B, *RUNS, 3 * 140 - 1, slack=e)


@pytest.mark.parametrize("burst", [1, 2, 3, 4])
@pytest.mark.parametrize("B", [1, 2, 5])
def test_queues_of_a_few(S, O, burst, B):  # noqa: F811
    """Bursts of a few requests, far enough apart that each burst is served before
    the next: the queue empties every time."""
    rng = np.random.default_rng(10 * B + burst)
    n = 24 * burst + 33
    o = np.stack([rng.choice([7, 7, 30], n), rng.integers(1, 50, n), np.full(n, 9)]).astype(np.int32)
    p = np.zeros_like(o)
    a = np.tile((np.arange(n) // burst * 50 * burst).astype(np.int32), (3, 1))
    for kv in (50, 120, INF):
        run_both(S, O, a, p, o, B, *RUNS, kv)
