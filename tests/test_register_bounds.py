"""Launch bounds that a block can have: the compiler divides the register file by them, so a bound above the
1024 threads of a block holds a kernel to half its registers.  The four-point snapshot transforms, bound at
2048 threads, were held to 32 registers and spilled; read from the compiler's own report (no GPU needed)."""
import os
import re
import subprocess

from paper_1808_05168_gb300 import build


def test_four_point_transforms_do_not_spill(tmp_path):
    cmd = [build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                                         "-Xptxas", "-v", "-cubin", os.path.join(build.CSRC, "lb_diag.cu"), "-o",
                                         str(tmp_path / "lb_diag.cubin")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    seen = re.findall(r"Function properties for \S*ps_(rows|cols)_kernelILi4E.*?(\d+) bytes spill stores.*?Used (\d+) registers",
                      r.stderr, re.S)
    assert sorted(k for k, _, _ in seen) == ["cols", "rows"]
    for _, spilled, regs in seen:
        assert int(spilled) == 0 and int(regs) <= 65536 // 1024
