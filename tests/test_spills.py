"""Registers that the row kernels' residency depends on, and spills where a kernel
has no other path."""
import functools
import importlib
import os
import re
import subprocess

import pytest


@pytest.fixture(scope="module")
def ptxas(tmp_path_factory):
    """file -> {kernel: (bytes spilled, registers)}"""
    build = importlib.import_module("paper_2602_05686_gb300.build")
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")

    @functools.lru_cache
    def get(name):
        r = subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, "-Xptxas", "-v", "-c",
                            os.path.join(build.CSRC, name + ".cu"), "-o",
                            str(tmp_path_factory.mktemp("o") / "v.o")], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return {k: (int(b), int(n)) for k, b, n in
                re.findall(r"Function properties for (\S+)\n\s*\d+ bytes stack frame, (\d+) bytes spill stores[^\n]*\n"
                           r"[^\n]*Used (\d+) registers", r.stderr)}
    return get


def test_sell_rows_spill_nothing(ptxas):
    # k_vc_*<T, 0> and <T, -2>: one and two lanes per SELL row
    sell = {k: v for k, v in ptxas("vcycle").items() if re.search(r"k_vc_\w+I[df]Li(0|n2)E", k)}
    assert len(sell) == 20
    assert not any(b for b, _ in sell.values()), sell


def test_group_rows_leave_room_for_four_blocks(ptxas):
    (spilled, regs), = [v for k, v in ptxas("group").items() if "k_g_matId" in k]
    assert spilled == 0 and regs <= 64


def test_outer_product_keeps_eight_blocks(ptxas):
    # 65536 registers / (8 x 256 threads)
    regs = [n for k, (_, n) in ptxas("vcycle").items() if "k_sell_spmv_dot" in k]
    assert len(regs) == 2 and max(regs) <= 32
