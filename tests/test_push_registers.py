"""The FP32 2D push kernels hold their particles in registers: what is asked for ahead of the tile must not spill
(order 3 lost 20 % of a small push to that)."""
import os
import re
import subprocess

from paper_1502_01376_gb300 import build


def test_fp32_push_does_not_spill(tmp_path):
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, "push.cu"),
                        "-o", str(tmp_path / "push.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = 0
    for name, stores in re.findall(r"Function properties for (\S+)\s+\d+ bytes stack frame, (\d+) bytes spill stores", r.stderr):
        if "k_push2dIf" in name:                    # k_push2d<float, ...>
            found += 1
            assert stores == "0", (name, stores)
    assert found == 6, r.stderr
