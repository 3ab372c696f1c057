"""The float64 kernels of the Krylov loops hold nothing in local memory.

Read from the compiler's own report of the build (-Xptxas -v).  Steps whose BiCGStab product
spilled its registers under a cap of blocks per SM raised "misaligned address".
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_float64_loop_kernels_do_not_spill():
    from paper_1602_03643_gb300 import build
    try:
        build.build()
    except RuntimeError as e:
        pytest.skip(str(e))
    path = os.path.join(ROOT, "paper_1602_03643_gb300", "_build", "ptxas.log")
    name, seen, bad = None, 0, []
    for line in open(path):
        m = re.search(r"Compiling entry function '(\S+)'", line)
        if m:
            name = m.group(1)
        m = re.search(r"(\d+) bytes stack frame", line)
        if m and name and "4Fp64" in name and re.search(r"\d+k_(bicg|pcg|amg_cg|mass|scalar)_", name):
            seen += 1
            if int(m.group(1)):
                bad.append((name, int(m.group(1))))
            name = None
    assert seen >= 40
    assert not bad, bad
