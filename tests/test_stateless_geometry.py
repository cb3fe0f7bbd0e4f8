"""Launch geometry of the stateless similarity calls, checked on the host (no GPU) by the C++ program
stateless_geometry.cu, linked against the built library."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_chunks_of_a_single_pair(tmp_path):
    from paper_2412_14671_gb300 import build

    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("nvcc missing")
    lib = build.build()
    exe = str(tmp_path / "stateless_geometry")
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "stateless_geometry.cu"), "-L", os.path.dirname(lib), "-lmuster",
                    "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", exe], check=True)
    # no device, so that the SM count is GB300's wherever this runs
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0 and "GEOMETRY-OK" in r.stdout, r.stdout + r.stderr
    assert int(r.stdout.split()[-1]) == 18**3 * 10
