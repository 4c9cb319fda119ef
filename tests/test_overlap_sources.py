"""The diagnostics kernels that may start before the launch before them has ended: none takes a parameter as
__restrict__, which with const would let the compiler read what that launch writes before the wait.  Read from
the source (no GPU needed), since a compiler that makes no use of it shows nothing."""
import os
import re

from paper_1808_05168_gb300 import build


def test_overlapping_diagnostics_take_plain_pointers():
    with open(os.path.join(build.CSRC, "lb_diag.cu")) as f:
        src = f.read()
    kernels = re.findall(r"__global__ void (?:__launch_bounds__\([^)]*\) )?(\w+)\(([^)]*)\) \{(.*?)\n\}", src, re.S)
    waiting = {name: params for name, params, body in kernels if "wait_for_previous_grid()" in body}
    assert set(waiting) == {"sf_rows_kernel", "sf_cols_kernel", "sample_tail_kernel"}
    for name, params in waiting.items():
        assert "__restrict__" not in params, name
