"""max_steps over its whole range: a guard that no run can reach is no guard."""
import subprocess

import numpy as np
import pytest

from conftest import cuda_available
from test_parity_gpu import INF, O, S, run_both  # noqa: F401  (fixtures)

PROG = r"""
#include <cstdio>
#include "sim_internal.cuh"
int main() {
    const int64_t top = INT32_MAX;
    const int64_t given[] = {1, 2, 1000, top - 2, top - 1, top, top + 1, (int64_t)1 << 40, INT64_MAX - 1, INT64_MAX};
    for (int64_t m : given) {
        const int32_t g = isjl::step_guard(m);
        if (g < 1 || (m < top ? g != m + 1 : g != top)) { printf("%lld: %d\n", (long long)m, g); return 1; }
    }
    puts("checked");
    return 0;
}
"""


def test_the_guard_step_of_every_bound(tmp_path):
    """The first step not to be served, max_steps + 1, where it is a step number."""
    from paper_2608_02244_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    src, exe = tmp_path / "guard.cu", tmp_path / "guard"
    src.write_text(PROG)
    subprocess.run([nvcc, str(src), "-o", str(exe)] + build._flags(False), check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "checked\n"


@pytest.mark.gpu
@pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("copies", [1, 4000])                 # a warp and a thread per task
@pytest.mark.parametrize("max_steps", [2**31 - 2, 2**31 - 1, 2**31, 2**63 - 2, 2**63 - 1])
def test_bounds_that_no_run_reaches(S, O, max_steps, copies):  # noqa: F811
    """The same results as without a bound; with predictions, where the default
    bound can end a run, the runs that it ends are finished."""
    rng = np.random.default_rng(6)
    o = np.tile(rng.integers(1, 60, (1, 12)), (copies, 1)).astype(np.int32)
    a = np.tile(np.sort(rng.integers(0, 90, (1, 12)), axis=1), (copies, 1)).astype(np.int32)
    z = np.zeros_like(o)
    pols, ds = ["fcfs", "ljf", "sjf", "isjl", "isjl", "isjl_beta"], [0, 0, 0, 5, INF, 9]
    res = run_both(S, O, a, z, o, 3, pols, ds, 100, max_steps=max_steps)
    free = run_both(S, O, a, z, o, 3, pols, ds, 100, check=False)
    assert (res["records"]["status"] == 0).all() and res["records"].tobytes() == free["records"].tobytes()
    o = np.tile(np.array([[1, 8, 3, 2, 40, 41]], np.int32), (copies, 1))
    slack = np.tile(np.array([[5, 5, 3, 4, 3, 1]], np.int32), (copies, 1))
    z = np.zeros_like(o)
    args = (z, z, o, 3, ["isjl_beta"] * 2 + ["isjl"], [9, 9, 9], 48)
    assert (run_both(S, O, *args, slack=slack)["records"]["status"] == S.ISJL_ERR_STEP_LIMIT).any()
    res = run_both(S, O, *args, slack=slack, max_steps=max_steps)
    assert (res["records"]["status"] == 0).all() and (res["completion"] >= 0).all()


@pytest.mark.gpu
@pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("copies", [1, 4000])                 # a warp and a thread per task
@pytest.mark.parametrize("max_steps", [0, 2**31 - 1])
def test_idling_at_the_end_of_the_step_range(S, max_steps, copies):  # noqa: F811
    """Predictions leave o_1's delay idle: packs planned with 2,000 tokens are done
    after two, and o_1 waits 1,000 steps.  The same requests at step 0 and at the
    last arrival that is accepted (sum o + max arrival = 2^30 - 2): every step is
    the same number of steps later, under the default bound (which ends the run in
    that idle time) and under one that no run reaches."""
    o = np.ones((copies, 4), np.int32)
    slack = np.tile(np.array([[4999, 3999, 999, 999]], np.int32), (copies, 1))
    z = np.zeros_like(o)
    late = 2**30 - 2 - int(o[0].sum())
    pols, ds = ["isjl", "isjl_beta", "isjl", "sjf"], [1000, 1000, INF, 0]
    sm = S.Simulator(copies, o.shape[1], 2, max_steps=max_steps)
    try:
        early = sm.sweep(z, z, o, pols, ds, INF, per_request=True, slack=slack)
        res = sm.sweep(z + late, z, o, pols, ds, INF, per_request=True, slack=slack)
    finally:
        sm.close()
    assert (early["records"]["status"][0] == (0 if max_steps else S.ISJL_ERR_STEP_LIMIT)).all()
    assert max_steps == 0 or (early["records"]["T_make"][0] > 1000).all()
    for f in ("status", "T_busy", "O", "Q", "W", "E", "token_adv", "sum_extent", "max_extent", "violations",
              "peak_kv", "peak_batch"):
        np.testing.assert_array_equal(res["records"][f], early["records"][f], err_msg=f)
    for f in ("start", "completion"):
        np.testing.assert_array_equal(res[f], np.where(early[f] < 0, -1, early[f] + late), err_msg=f)
