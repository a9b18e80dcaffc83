"""The autotuner's choice of a schedule from its samples (CPU, nvcc): the fastest
where a product stands alone, the default inside an eigensolver unless another
is faster by more than the samples differ.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "cuda_backend.h"
using namespace tns;
int main() {
  const float tie[3] = {1.1031f, 0.9180f, 0.9078f}, tie2[3] = {1.1145f, 0.9089f, 0.9144f};  // two runs of one list
  const float clear[3] = {5.3930f, 4.7345f, 4.2192f};
  const float low[4] = {0.4685f, 0.3973f, 0.3475f, 0.7244f}, far[4] = {0.5f, 0.4f, 0.3f, 0.5f};
  std::printf("%d %d %d ", pick_variant(tie, 3, kSteadyFp64), pick_variant(tie2, 3, kSteadyFp64),
              pick_variant(clear, 3, kSteadyFp64));
  std::printf("%d %d ", pick_variant(low, 4, kSteady), pick_variant(far, 4, kSteady));
  std::printf("%d %d %d\n", pick_variant(tie, 3, 1.0), pick_variant(tie2, 3, 1.0), pick_variant(low, 4, 1.0));
}
"""


def test_choice(tmp_path):
    from paper_2305_05581_gb300 import build as b
    nv = b.nvcc()
    if not (os.path.exists(nv) or shutil.which(nv)):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "choice.cu", tmp_path / "choice"
    src.write_text(SRC)
    subprocess.check_call([nv, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", b.CSRC,
                           "-o", str(exe), str(src)])
    assert subprocess.check_output([str(exe)], text=True).split() == ["1", "1", "2", "1", "2", "2", "1", "2"]
