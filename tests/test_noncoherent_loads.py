"""Kernels that may be on the SMs while the one ahead of them still writes (launch() in conef_internal.h) must not read its
results by ld.global.nc, which is for memory that nobody writes while the grid lives."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_08538_b200", "csrc")


def test_ldg_reads_tables_of_the_plan_only():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                text = re.sub(r"//.*", "", f.read())
            if "cudaLaunchCooperativeKernel" in text:   # (an ordinary launch: nothing ahead of it runs on)
                continue
            found += [(name, m.group(1)) for m in re.finditer(r"(?:__ldg|ld\.global\.nc)\w*\(?([^;]*)", text)]
    assert found and all(n == "conef_common.cuh" and arg.startswith("pfx + ") for n, arg in found), found
