"""The order that launches as programmatic dependents rely on, read off the
kernels' source: a kernel that waits for the launch before it does so before
any exit and before it allocates tensor memory, and one that allocates lets
the next launch begin only after that.  (A kernel that held tensor memory while
it waited could keep the columns from CTAs it waits for.  Nothing here runs.)"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_14317_gb300", "csrc")


def _kernels():
    """(name, body without comments) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        src = open(os.path.join(CSRC, f)).read()
        src = re.sub(r"//[^\n]*", "", src)
        src = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", src)
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\([^{;]*?\)\s*\{", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            yield pytest.param(src[m.end():i], id=m.group(1))


WAIT, BOTH, RELEASE, ALLOC = "grid_await();", "grid_wait();", "grid_release();", "tcgen05.alloc"


@pytest.mark.parametrize("body", list(_kernels()))
def test_wait_before_exit_and_allocation(body):
    waits = [i for i in (body.find(WAIT), body.find(BOTH)) if i >= 0]
    if not waits:   # launched plainly
        assert RELEASE not in body
        return
    first = min(waits)
    exits = [m.start() for m in re.finditer(r"\breturn;", body)]   # of the kernel: lambdas return values
    assert all(first < i for i in exits)
    if ALLOC in body:
        assert BOTH not in body
        assert first < body.find(ALLOC) < body.find(RELEASE)


def test_the_chained_kernels_are_seen():
    bodies = {p.id: p.values[0] for p in _kernels()}
    for k in ("eval_pipe_kernel", "eval_mixed_kernel"):
        assert WAIT in bodies[k] and ALLOC in bodies[k] and RELEASE in bodies[k]
    for k in ("eval_fx_kernel", "gj_update_kernel", "step_fp64_kernel", "null64_kernel", "sum_columns_kernel"):
        assert BOTH in bodies[k]


@pytest.mark.gpu
@pytest.mark.parametrize("p", [1, 300])
def test_evaluation_then_step(hpt, p):
    """A small mixed evaluation directly followed by steps of the same stream
    (both kernels allocate tensor memory): the bits of separate calls."""
    import torch

    import workloads as W

    s = W.laurent_system(70, 9, 6, -2, 2, 8, nnz=4)
    h = hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": W.random_alpha(5, 9, -1, 1).tolist(), "denom": 1}, 1)
    y, t = W.random_points(9, p, 9)
    yd, td = torch.from_numpy(y).to("cuda", torch.complex64), torch.from_numpy(t).cuda()
    y0 = torch.from_numpy(y).cuda()
    prm = hpt.Params(tol_accept=1e-2, eps0=1e-2)
    out = []
    for between in (torch.cuda.synchronize, lambda: None):
        st = h.new_state(p)
        for _ in range(3):
            h.paths_init(st, y0, prm)
            between()
            H = h.eval(yd, td)
            between()
            h.step(st, 2, prm)
            between()
        torch.cuda.synchronize()
        assert h.device_error() == 0
        out.append([a.clone() for a in H] + [st.arena.clone()])
    for a, b in zip(*out):
        assert torch.equal(a, b)
