"""Instances of few requests on the GPU against the oracle: the thread-per-task
simulation (up to 32 requests, many tasks) at the edges of its range and one
request beyond it, and the preparation kernels at the edges of their sizes."""
import numpy as np
import pytest

from conftest import cuda_available
from test_parity_gpu import INF, O, S, run_both  # noqa: F401  (fixtures)

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n", [1, 2, 7, 31, 32, 33])
@pytest.mark.parametrize("B", [1, 3, 31, 32, 40])
def test_many_small_instances(S, O, n, B):  # noqa: F811
    rng = np.random.default_rng(1000 * n + B)
    N = 4500                                    # x 7 runs: more than 10.6 waves of 2,432 warps
    o = rng.choice(np.array([1, 3, 3, 8, 21, 40], np.int32), (N, n)).astype(np.int32)
    p = rng.integers(0, 2, (N, n)).astype(np.int32)
    a = np.sort(rng.integers(0, 4 * n, (N, n)), axis=1).astype(np.int32)
    a[::2] = 0
    pols, ds = ["fcfs", "ljf", "sjf", "isjl", "isjl", "isjl", "isjl_beta"], [3, 0, 0, 0, 5, INF, 9]
    counts = rng.integers(0, n + 1, N).astype(np.int32)
    slack = rng.integers(0, 6, (N, n)).astype(np.int32)
    big = 48
    run_both(S, O, a, p, o, B, pols, ds, INF)
    run_both(S, O, a, p, o, B, pols, ds, big, counts=counts, slack=slack)
    run_both(S, O, a, p, o, B, pols, ds, 2 * big, max_steps=n + 9)


@pytest.mark.parametrize("copies", [1, 4000])                 # a warp and a thread per task
def test_step_bound_with_predictions(S, O, copies):  # noqa: F811
    """Predictions can leave o_1's delay idle, so that a run reaches the bound
    sum o + max arrival: status STEP_LIMIT, partial counters, -1 for the request
    still running.  Without prefilled outputs and through the binding."""
    o = np.tile(np.array([[1, 8, 3, 2, 40, 41]], np.int32), (copies, 1))
    slack = np.tile(np.array([[5, 5, 3, 4, 3, 1]], np.int32), (copies, 1))
    z = np.zeros_like(o)
    res = run_both(S, O, z, z, o, 3, ["isjl_beta"] * 2 + ["isjl"], [9, 9, 9], 48, slack=slack)
    assert (res["records"]["status"] == S.ISJL_ERR_STEP_LIMIT).any()
    assert (res["completion"] == -1).any()


@pytest.mark.parametrize("n", [31, 33, 127, 129, 256, 257, 512, 513, 1024, 1025, 4096, 4097, 8193])
def test_preparation_sizes(S, O, n):  # noqa: F811
    rng = np.random.default_rng(n)
    o = rng.choice(np.array([1, 2, 2, 255, 256, 257, 3000], np.int32), (3, n)).astype(np.int32)
    o[1] = rng.integers(1, 3000, n)
    p = np.zeros_like(o)
    a = np.zeros_like(o)
    counts = np.array([n, max(1, n - 1), n // 2], np.int32)
    run_both(S, O, a, p, o, 64, ["ljf", "sjf"], [0, 0], INF, counts=counts)
