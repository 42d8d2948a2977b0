"""The FP64 re-solve of flagged paths inside the FP32 solve's warps (GPU): one to
four flagged paths in a warp take different lane groups, with the same bits as
the path on its own."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _system(hpt, n):
    s = W.laurent_system(80 + n, n, 3 if n == 1 else 6, -2, 2, 8, nnz=min(n, 4))
    return hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": W.random_alpha(5, n, -1, 1).tolist(), "denom": 1}, 1)


@pytest.mark.parametrize("cond_max", [1.0, 10.0, 40.0, 200.0])
@pytest.mark.parametrize("n", [1, 4, 8, 9, 16, 17, 32])
def test_step_bits_do_not_depend_on_the_neighbours(hpt, n, cond_max):
    h = _system(hpt, n)
    p = 37
    y, t = W.random_points(n, p, n)
    prm = hpt.Params(cond_max=cond_max, tol_accept=1e-2)

    def run(sel):
        st = h.new_state(len(sel))
        st.y.copy_(torch.from_numpy(y[sel]).cuda())
        st.y_acc.copy_(st.y)
        st.tau.copy_(torch.from_numpy(np.log(0.3 + 0.7 * t[sel])))
        st.tau_acc.copy_(st.tau)
        st.dtau.fill_(0.01)
        st.accepts.fill_(1)
        h.step(st, 2, prm)
        return {k: v.numpy() for k, v in st.to_host().items()}

    together = run(np.arange(p))
    for q in range(p):
        alone = run(np.array([q]))
        for k, v in alone.items():
            assert np.array_equal(v[0], together[k][q], equal_nan=True), (q, k)


@pytest.mark.parametrize("cond_max", [1.0, 20.0, 200.0])
@pytest.mark.parametrize("n", [5, 12, 20, 24, 28])
def test_batch_bits_do_not_depend_on_the_neighbours(hpt, n, cond_max):
    h = _system(hpt, n)
    p = 19
    y = torch.from_numpy(W.random_points(n, p, n)[0]).cuda()
    prm = hpt.Params(cond_max=cond_max, tol_accept=1e-2, max_steps=12, eps0=1e-2)
    x, st, sp = hpt.Batch([h]).track(y.reshape(-1), [p], prm)
    b = hpt.Batch([h])
    for q in range(p):
        x1, st1, sp1 = b.track(y[q].contiguous(), [1], prm)
        assert torch.equal(st1, st[q:q + 1]) and torch.equal(sp1, sp[q:q + 1])
        assert np.array_equal(x1.cpu().numpy(), x.view(p, n)[q].cpu().numpy(), equal_nan=True)
