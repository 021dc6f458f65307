"""The coarse factor's square root and reciprocal are those of sqrt() and a
division, bit for bit."""
import importlib
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    build = importlib.import_module("paper_2602_05686_gb300.build")
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    out = tmp_path_factory.mktemp("pivot") / "pivot"
    r = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-O2", "-I", build.CSRC, os.path.join(HERE, "pivot.cu"), "-o",
                        str(out)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(out)


def run(exe, mode):
    r = subprocess.run([exe, mode], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)


def test_settled_from_starting_values_off_by_four_units(exe):
    run(exe, "host")


@pytest.mark.gpu
def test_on_the_gpu(exe):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    run(exe, "gpu")
