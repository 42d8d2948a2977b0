"""Launch limits (CPU): a kernel's dynamic shared-memory limit is a property of
the process, shared by all host threads, so no launch may set it to an amount
of its own."""
import os
import re

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
