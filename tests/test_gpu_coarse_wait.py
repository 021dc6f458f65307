"""The coarse factor's bounded waits: a launch whose waits run out ends by itself
with the error bit, and the GPU goes on."""
import importlib
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_waits_that_run_out_end_the_launch(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build = importlib.import_module("paper_2602_05686_gb300.build")
    build.build()
    exe = tmp_path / "wait"
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O2", "-I", os.path.join(build.ROOT, "include"), "-I",
                        build.CSRC, os.path.join(HERE, "coarse_wait.cu"), "-o", str(exe), "-L", build.OUT_DIR,
                        "-lsa_gb300", "-Xlinker", "-rpath=" + build.OUT_DIR], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr)
