"""The FP32 in-place odd step keeps its registers: its ring's code once spilled 56 bytes, which cost
steps of 450^2 to 512^2 cavities 4 percent."""
import os
import re
import subprocess

from paper_1708_07525_gb300 import build


def test_the_fp32_in_place_odd_step_does_not_spill(tmp_path):
    r = subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas=-v", "-c", os.path.join(build.CSRC, "lbm_k_f32.cu"),
                        "-o", str(tmp_path / "k.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found = re.findall(r"Compiling entry function '\w*step_aa_odd_fused_kernel\w*'.*?(\d+) bytes spill stores", r.stderr, re.S)
    assert found and set(found) == {"0"}
