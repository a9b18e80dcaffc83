"""Resource budgets of the FP64 product kernels, from the assembler's own report
(`nvcc -Xptxas -v`, CPU only), as test_kernel_resources.py holds the
tensor-core form's: registers within the SM's 64 K at the designed number of
resident CTAs, and no spills.

  k_tasks_im, classes of 1, 2, 4 warps   12, 4, 2 CTAs per SM   -> <= 168, 255, 255 registers
  k_tasks_fp64 and k_tasks_fp64_failed   512 threads per SM     -> <= 128
"""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_05581_gb300", "csrc")


@pytest.fixture(scope="module")
def report():
    from paper_2305_05581_gb300 import build as b
    nv = b.nvcc()
    if not (os.path.exists(nv) or shutil.which(nv)):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.join(ROOT, "_build"), exist_ok=True)
    kernels, name = {}, None
    for src in ("fp64_digits.cu", "kernels.cu"):
        obj = os.path.join(ROOT, "_build", src + "_resources.o")
        r = subprocess.run([nv] + b.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                                            "-Xptxas", "-v", "-c", os.path.join(CSRC, src), "-o", obj],
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
        for line in r.stderr.splitlines():
            m = re.search(r"Compiling entry function '([^']+)'", line)
            if m:
                name = m.group(1)
                kernels[name] = {}
            m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
            if m and name:
                kernels[name].setdefault("spill", int(m.group(1)) + int(m.group(2)))
            m = re.search(r"Used (\d+) registers", line)
            if m and name:
                kernels[name].setdefault("regs", int(m.group(1)))
    return kernels


@pytest.mark.parametrize("stem,count,budget", [("k_tasks_imI.*ImCfgILi1E", 1, 168), ("k_tasks_imI.*ImCfgILi2E", 1, 255),
                                               ("k_tasks_imI.*ImCfgILi4E", 1, 255), ("k_tasks_fp64ILi", 4, 128),
                                               ("k_tasks_fp64_failedILi", 3, 128)])
def test_registers_fit_the_designed_residency(report, stem, count, budget):
    hits = {n: k for n, k in report.items() if re.search(stem, n)}
    assert len(hits) == count, (stem, sorted(hits))
    for n, k in hits.items():
        assert k["regs"] <= budget and k["spill"] == 0, (n, k)
