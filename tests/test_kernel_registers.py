"""Registers of the window-sum kernels (no GPU): every window and similarity is cut for the CTAs per SM that its own
shared memory allows, so none of the 40 instantiations spills to local memory (beyond two words of the smallest
window, whose registers are the limit)."""
import os
import re
import shutil
import subprocess

import pytest


def test_window_sum_kernels_do_not_spill(tmp_path):
    from paper_2412_14671_gb300 import build

    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("nvcc missing")
    r = subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, "sim_kernels.cu"),
                        "-o", str(tmp_path / "sim.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    log = r.stdout + r.stderr
    found = re.findall(r"Compiling entry function '\S*k_sim_(fwd|bwd)ILi(\d)ELi(\d)ELb(\d)\S*'.*?(\d+) bytes spill stores",
                       log, re.S)
    assert len(found) == 40
    for which, radius, kind, staged, spilled in found:
        assert int(spilled) <= (8 if radius == "1" else 0), (which, radius, kind, staged, spilled)
