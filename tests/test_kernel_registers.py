"""Registers and spills of direct step kernels, as the compiler reports them: forms
whose speed hangs on how many blocks share an SM.  They grew unnoticed when a kernel
argument moved and a call was put behind the row loop."""
import os
import re
import shutil
import subprocess

import pytest

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_00530_gb300")
NVCC = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
# (kernel, closure, storage, vector, noise form): bytes spilled, registers at most.  65536
# registers, allotted in eights a thread, hold that many blocks of 128 threads: 6 at 80, 5 at
# 96, 7 at 72, 8 at 64.
PASSIVE, CIL, F32, F16 = 0, 2, 0, 1
LIMITS = {("step_kernel", CIL, F32, 4, 1): (0, 80), ("step_kernel", PASSIVE, F32, 4, 1): (0, 80),
          ("step_kernel", PASSIVE, F16, 4, 0): (0, 72), ("step_kernel", CIL, F16, 4, 1): (68, 80),
          ("step_kernel_q7", CIL, F32, 4, 1): (0, 96), ("step_kernel_q7", PASSIVE, F32, 4, 1): (0, 96),
          ("step_kernel_q7", CIL, F32, 2, 1): (0, 64), ("step_kernel_q7", PASSIVE, F16, 4, 0): (0, 64)}


@pytest.mark.skipif(NVCC is None, reason="no nvcc")
def test_direct_kernels_keep_their_registers(tmp_path):
    src = tmp_path / "forms.cu"
    src.write_text('#include "lbm_step_q7.cuh"\n' + "".join(
        f"template __global__ void lbm::{k}<{m}, {st}, {v}, false, {n}, false>(const lbm::StepArgs);\n"
        for k, m, st, v, n in LIMITS))
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-Xptxas=-v",
                        "-I", os.path.join(PKG, "csrc"), "-c", str(src), "-o", str(tmp_path / "forms.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    got = {}
    for block in r.stderr.split("Compiling entry function")[1:]:
        name = re.search(r"(step_kernel(?:_q7)?)ILi(\d)ELi(\d)ELi(\d)ELb0ELi(\d)ELb0E", block)
        if name:
            got[(name[1], *map(int, name.groups()[1:]))] = (int(re.search(r"(\d+) bytes spill stores", block)[1]),
                                                           int(re.search(r"Used (\d+) registers", block)[1]))
    assert set(got) == set(LIMITS)
    over = {k: v for k, v in got.items() if v[0] > LIMITS[k][0] or v[1] > LIMITS[k][1]}
    assert not over, over
