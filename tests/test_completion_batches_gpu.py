"""Batches of completions on the GPU against the oracle: runs whose queue head
waits for KV or a slot, at the sizes and lengths where a batch has to stop or to
fall back (more than 32 completions at one step, requests shorter than the
batch, one slot, every row count, slack, a step guard inside a batch)."""
import numpy as np
import pytest

from conftest import cuda_available
from test_parity_gpu import INF, O, S, run_both  # noqa: F401  (fixtures)

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]

POLICIES = ["fcfs", "isjl", "sjf"]


def lengths(rng, kind, shape):
    if kind == "ties":                      # whole batches complete at one step
        return rng.choice(np.array([40, 40, 40, 41], np.int32), shape).astype(np.int32)
    if kind == "short":                     # many requests end before the batch they start in
        return np.where(rng.random(shape) < 0.5, rng.integers(1, 4, shape), rng.integers(100, 900, shape)).astype(
            np.int32)
    if kind == "long":                      # lengths up to the limit
        return np.minimum(rng.pareto(1.1, shape) * 300 + 1, 65_535).astype(np.int32)
    return rng.integers(1, 2000, shape).astype(np.int32)


@pytest.mark.parametrize("policy", POLICIES)
@pytest.mark.parametrize("kind", ["ties", "short", "long", "mixed"])
@pytest.mark.parametrize("B", [1, 5, 32, 33, 64, 128, 200, 512])
def test_batches_of_completions(S, O, policy, kind, B):  # noqa: F811
    rng = np.random.default_rng(100 + B)
    n = 700
    o = lengths(rng, kind, (3, n))
    p = np.zeros_like(o)
    a = np.zeros_like(o)
    a[1] = np.sort(rng.integers(0, 300, n))
    a[2] = np.sort(rng.integers(0, 20_000, n))          # queue empty now and then
    big = int(o.max())
    for kv, slack, ms in [(INF, None, 0), (max(big, int(o.mean() * B * 0.6)), None, 0),
                          (big + 40, rng.integers(0, 40, o.shape).astype(np.int32), 0), (big * 3, None, 997)]:
        if slack is not None:
            o = np.minimum(o, 65_535 - 40)
        run_both(S, O, a, p, o, B, [policy] * 2, [50, INF], kv, slack=slack, max_steps=ms)


def test_budgets_around_the_longest_length(S, O):  # noqa: F811
    """A budget of 65,535 or more never plans and never shuts the gate and has
    a body of its own; 65,534 still can, with a request of 65,535 tokens."""
    rng = np.random.default_rng(9)
    o = lengths(rng, "long", (4, 60))
    o[:, :3] = 65_535
    o[1, 3:6] = 65_534
    p = np.zeros_like(o)
    a = np.zeros_like(o)
    a[2:] = np.sort(rng.integers(0, 90_000, (2, 60)), axis=1)
    for B in (2, 5, 40):
        for pol in ("isjl", "isjl_beta"):
            run_both(S, O, a, p, o, B, [pol] * 4, [65_533, 65_534, 65_535, INF], INF)
            run_both(S, O, a, p, o, B, [pol] * 4, [65_533, 65_534, 65_535, INF], 150_000)


@pytest.mark.parametrize("policy, n", [("sjf", 260), ("sjf", 99), ("sjf", 100), ("fcfs", 260), ("fcfs", 99), ("fcfs", 100)])
@pytest.mark.parametrize("kv", [INF, 30_000, 6_000])
@pytest.mark.parametrize("B", [3, 7, 8, 15, 16, 32, 100])
def test_both_sides_of_the_queue_rules(S, O, policy, n, kv, B):  # noqa: F811
    """FCFS and SJF have batches from 100 requests on where their tokens are more
    than some times what the slots or the KV serve until the last arrival: last
    arrivals around each line, few and many lengths, and more than 32 requests of
    the shortest one."""
    rng = np.random.default_rng(17 + B)
    o = np.stack([rng.integers(1, 900, n), rng.integers(1, 900, n), rng.choice([90, 91, 92], n),
                  np.full(n, 250), rng.integers(1, 5, n) * 100, rng.integers(1, 40, n)]).astype(np.int32)
    O_ = o.sum(axis=1, dtype=np.int64)
    fit = kv * n // O_
    served = np.minimum(B, fit)
    line = O_ // (3 * served) if policy == "sjf" else np.where(fit < B, 3 * O_ // (2 * served), O_ // served)
    p = np.zeros_like(o)
    for last in (line - 1, line, line + 1, line // 3):
        a = np.sort(rng.random((6, n)) * last[:, None], axis=1).astype(np.int32)
        a[:, -1] = last
        run_both(S, O, a, p, o, B, [policy], [0], kv)
