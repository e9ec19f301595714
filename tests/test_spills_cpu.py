"""Registers of the tensor-core kernels, as the compiler reports them (no GPU needed).

Their row threads hold a whole tile row, so the kernels sit at the edge of their register budget, and a field or a loop
invariant more anywhere in them, in code that all roles share, turns into spills in the row loop."""
import os
import re
import subprocess

import pytest

from paper_2604_16429_b200 import build as mbuild

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

# most bytes a thread may spill (stores, loads)
LIMITS = {"bwd_dkdv_tc.cu": (40, 48), "bwd_dq_tc.cu": (0, 0), "fwd_tc.cu": (0, 0)}


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
@pytest.mark.parametrize("source", sorted(LIMITS))
def test_tensor_core_kernels_do_not_spill_more(source, tmp_path):
    log = subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo", "-Xptxas", "-v",
                          "-Xcompiler", "-fPIC", "-I", mbuild.INCLUDE, "-I", mbuild.CSRC, "-c", os.path.join(mbuild.CSRC, source),
                          "-o", str(tmp_path / "out.o")], check=True, capture_output=True, text=True).stderr
    found = re.findall(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", log, re.S)
    spills = {name: (int(st), int(ld)) for name, st, ld in found if "_tc_kernel" in name}
    assert len(spills) >= 4, log
    for name, (st, ld) in spills.items():
        assert st <= LIMITS[source][0] and ld <= LIMITS[source][1], (name, st, ld)
