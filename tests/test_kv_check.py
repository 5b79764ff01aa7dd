"""A run whose reserved KV went beyond the cap has status INTERNAL, whichever
kernel simulated it, although every start is checked before it."""
import os
import re
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2608_02244_gb300", "csrc")
PROG = r"""
#include <cstdio>
#include "sim_internal.cuh"
int main() {
    const int64_t caps[] = {1, 300, ISJL_KV_INF};
    for (int64_t cap : caps)
        for (int64_t over = -1; over <= 1; ++over) {
            if (cap + over > ISJL_KV_INF) continue;
            for (int64_t status : {ISJL_OK, ISJL_ERR_STEP_LIMIT})
                if (isjl::checked_status(status, (int32_t)(cap + over), cap) != (over > 0 ? ISJL_ERR_INTERNAL : status))
                    return 1;
        }
    puts("checked");
    return 0;
}
"""


def test_a_peak_beyond_the_cap_is_an_internal_error(tmp_path):
    from paper_2608_02244_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(PROG)
    subprocess.run([nvcc, str(src), "-o", str(exe)] + build._flags(False), check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "checked\n"


@pytest.mark.parametrize("source", ["sim_kernel.cu", "tiny_kernel.cu"])
def test_every_record_is_stored_after_the_check(source):
    with open(os.path.join(CSRC, source)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert text.count("store_record(") == 1
    assert 0 < text.find("checked_status(") < text.find("store_record(")
