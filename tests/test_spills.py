"""Registers of the row kernels whose only path would pay for spills."""
import importlib
import os
import re
import subprocess

import pytest


def test_sell_rows_spill_nothing(tmp_path):
    build = importlib.import_module("paper_2602_05686_gb300.build")
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    r = subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, "-Xptxas", "-v", "-c",
                        os.path.join(build.CSRC, "vcycle.cu"), "-o", str(tmp_path / "v.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    spills = dict(re.findall(r"Function properties for (\S+)\n\s*\d+ bytes stack frame, (\d+) bytes spill stores", r.stderr))
    # k_vc_*<T, 0> and <T, -2>: one and two lanes per SELL row
    sell = {k: int(v) for k, v in spills.items() if re.search(r"k_vc_\w+I[df]Li(0|n2)E", k)}
    assert len(sell) == 20
    assert not any(sell.values()), sell
