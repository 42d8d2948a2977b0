"""Handles of their own on host threads of their own (GPU): the launch limits
of a kernel are process-wide, so threads whose launches of the same kernel need
different amounts of shared memory must not take each other's."""
import threading

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("calls", ["step", "eval"])
def test_threads_with_different_shared_memory(hpt, calls):
    # step: the FP32 solve needs 53 KB a block at n = 28, 70 KB at n = 32;
    # eval: the mixed evaluation's buffers grow with n and the support
    shapes = [(28, 8), (32, 8)] if calls == "step" else [(18, 6), (24, 60)]
    p, reps = 4, 4000
    handles, errors, results = [], [], {}
    for n, m in shapes * 4:
        s = W.laurent_system(n, n, m, -2, 2, 8, nnz=4)
        handles.append(hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": [0] * n, "denom": 1}, 1))

    def work(i, h):
        try:
            y, t = W.random_points(h.n, p, h.n)
            y0, td = torch.from_numpy(y).cuda(), torch.from_numpy(t).cuda()
            stream = torch.cuda.Stream()
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                if calls == "step":
                    prm = hpt.Params(tol_accept=1e-2, eps0=1e-2)
                    st = h.new_state(p)
                    h.paths_init(st, y0, prm)
                    for _ in range(reps):
                        h.step(st, 1, prm)
                    results[i] = [st.arena]
                else:
                    yc = y0.to(torch.complex64)
                    out = h.eval(yc, td)
                    for _ in range(reps):
                        h.eval(yc, td, out=out)
                    results[i] = list(out)
                stream.synchronize()
        except Exception as e:   # noqa: BLE001 - reported by the main thread
            errors.append((h.n, repr(e)))

    threads = [threading.Thread(target=work, args=a) for a in enumerate(handles)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for i in range(6):   # the same work on several threads
        for a, b in zip(results[i], results[i + 2]):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=a.dtype != torch.uint8)
