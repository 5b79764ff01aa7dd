"""The per-run summaries: every field of isjl_summary against numpy over the
records of the same call, at instance counts where some warps or whole blocks of
the reduction have no record, one, or one more than others; and, in the source,
the order of the barriers around its stores into another block."""
import glob
import os
import re

import numpy as np
import pytest

from conftest import ROOT, cuda_available

INF = 2**31 - 1
SUMS = ("T_make", "T_busy", "O", "Q", "W", "E", "token_adv", "sum_completion", "sum_latency", "sum_extent",
        "violations", "kv_violations")
COSTS = ("c_T", "tau_Q", "tau_E", "cost", "revenue", "profit")


def kernels(text):
    """(name, body) of every __global__ function of a CUDA source, comments removed."""
    text = re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)
    for m in re.finditer(r"__global__\s[^;{]*?\b(\w+)\s*\([^;{()]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


def test_remote_shared_memory_only_after_a_cluster_barrier():
    """A block may touch another block's shared memory only once that block has
    started: a kernel that does so waits on a cluster barrier first, and again
    after its last access, so that no block's memory is gone too early."""
    found = 0
    for path in glob.glob(os.path.join(ROOT, "paper_2608_02244_gb300", "csrc", "*.cu")):
        with open(path) as f:
            for name, body in kernels(f.read()):
                access = [m.start() for m in re.finditer(r"(?:ld|st|atom|red)(?:\.\w+)*\.shared::cluster", body)]
                if not access:
                    continue
                found += 1
                arrive = [m.start() for m in re.finditer(r"barrier\.cluster\.arrive", body)]
                wait = [m.start() for m in re.finditer(r"barrier\.cluster\.wait", body)]
                assert len(arrive) == len(wait) == 2, name
                assert arrive[0] < wait[0] < access[0] <= access[-1] < arrive[1] < wait[1], name
    assert found == 1


@pytest.mark.gpu
@pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("n_inst", [1, 7, 16, 17, 127, 128, 129, 1023, 1025])
def test_every_field_against_the_records(n_inst):
    """128 warps share a run's records, 16 a block: the record of instance i
    belongs to block (i % 128) / 16.  Failing instances carry different statuses,
    and the first of them lies in another block than the one that reports."""
    from paper_2608_02244_gb300 import sim
    rng = np.random.default_rng(n_inst)
    n = 9
    a = np.sort(rng.integers(0, 40, (n_inst, n)), axis=1).astype(np.int32)
    p = rng.integers(0, 9, (n_inst, n)).astype(np.int32)
    o = rng.integers(1, 90, (n_inst, n)).astype(np.int32)
    policies, deltas = ["fcfs", "ljf", "isjl", "isjl", "sjf", "isjl_beta"], [3, 0, 0, 12, 7, 12]
    kv = 300
    for bad in ([], [n_inst - 1], [i for i in (120, 128, 5, 1000) if i < n_inst]):
        for max_steps in (0, 170):                       # the guard stops some runs and not others
            pb, ab = p.copy(), a.copy()
            for j, i in enumerate(bad):
                if j % 2:
                    ab[i] = ab[i][::-1] + np.arange(n, 0, -1)          # decreasing arrivals: invalid
                else:
                    pb[i, 4] = kv                                      # can never start: infeasible
            S = sim.Simulator(n_inst, n, 3, max_steps=max_steps)
            try:
                res = S.sweep(ab, pb, o, policies, deltas, kv)
            finally:
                S.close()
            for r, (pol, d) in enumerate(zip(policies, deltas)):
                R, s = res["records"][r], res["summaries"][r]
                assert (R["status"][bad] != 0).all()
                failed = np.flatnonzero(R["status"])
                assert s["status"] == (R["status"][failed[0]] if failed.size else 0)
                assert (s["policy"], s["delta"], s["kv_cap"]) == (sim.POLICY[pol], d, kv)
                assert s["n_instances"] == n_inst and s["n_ok"] == n_inst - failed.size
                for f in SUMS:
                    assert s[f] == int(R[f].sum()), f
                assert s["max_extent"] == int(R["max_extent"].max())
                for f in COSTS:                          # two orders of one sum of n terms
                    assert abs(s[f] - R[f].sum()) <= 2 * n_inst * 2.0**-53 * np.abs(R[f]).sum(), f
