"""Launch limits (CPU): a kernel's dynamic shared-memory limit is a property of
the process, shared by all host threads, so no launch may set it to an amount
of its own.  Refused launches (GPU): reported once."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_14317_gb300", "csrc")


def test_one_limit_per_kernel():
    """Every limit goes through allow_smem, whose value is a template argument
    and so cannot depend on the launch."""
    calls = []
    for f in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        calls += [(f, m) for m in re.findall(r"cudaFuncSetAttribute\([^;]*", src)]
    assert [f for f, _ in calls] == ["hpt_internal.h"]
    assert "kMost" in calls[0][1]
    assert re.search(r"template <int kMost, typename K>\s+inline cudaError_t allow_smem",
                     open(os.path.join(CSRC, "hpt_internal.h")).read())


@pytest.mark.gpu
def test_a_refused_launch_is_reported_once(tmp_path):
    """A launch that the runtime refuses (1 GB of shared memory a block) returns
    its error and leaves none behind for the next launch's check."""
    src = tmp_path / "refused.cu"
    src.write_text(r"""
#include <cstdio>
#include "hpt_internal.h"
__global__ void nothing(int) {}
int main() {
  if (cudaFree(0) != cudaSuccess) return 2;
  const cudaError_t e = hpt::launch_chained(nothing, 1, 32, (size_t)1 << 30, 0, true, 1);
  const cudaError_t left = cudaGetLastError();
  nothing<<<1, 32>>>(1);
  const cudaError_t next = cudaGetLastError();
  printf("%d %d %d\n", e != cudaSuccess, (int)left, (int)next);
  return cudaDeviceSynchronize() != cudaSuccess;
}
""")
    from paper_2111_14317_gb300 import build
    exe = tmp_path / "refused"
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o",
                    str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.split() == ["1", "0", "0"], (r.returncode, r.stdout)
