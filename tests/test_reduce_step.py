"""The scalar step that follows a fixed-order reduction reads the sums it has and
no others: the device code, compiled for the host, on sums that end at an
unreadable page."""
import importlib
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_step_reads_only_its_sums(tmp_path):
    build = importlib.import_module("paper_2602_05686_gb300.build")  # (the package exports a function of that name)
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = tmp_path / "step"
    r = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC,
                        os.path.join(HERE, "host_reduce_step.cu"), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stderr)


def test_wide_finish_sums_the_columns_that_were_written():
    """a launch for k columns of partial sums takes k values, a warp each: the
    operator product writes no others"""
    import re
    build = importlib.import_module("paper_2602_05686_gb300.build")
    src = open(os.path.join(build.CSRC, "solve.cu")).read()
    body = src[src.index("int launch_fin_wide("):]
    body = body[:body.index("\n}")]
    assert body.count("launch_pdl(") == 4
    for k in (0, 2, 4, 8):
        assert re.search(rf"case {k}: launch_pdl\(k_fin_wide<{k or 1}>, 32, {32 * (k or 1)}, 0, st, part, np, "
                         rf"{'np' if k else '0'}, fin\); break;", body), k
    assert "default: return SA_ERR_INVALID_ARG;" in body
