"""The FP64 solve's lane-group shapes (GPU).  Few paths take 32 lanes each,
more 16, many 8 (n <= 16) or 16 lanes; an entry's arithmetic does not depend on
the shape, so the same paths give the same bits in a small and in a large
call.  (The small shape's step is compared with the oracle in
test_gpu_step.py, n = 1 .. 32.)"""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 24, 31, 32])
def test_shapes_give_the_same_bits(hpt, n):
    s = W.laurent_system(40 + n, n, 3 if n == 1 else 5, -2, 2, 8, nnz=min(n, 4))
    alpha = W.random_alpha(3, n, -1, 1)
    h = hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": alpha.tolist(), "denom": 1}, 0)
    big, mid, small = 4900, 2500, 37   # 8 or 16 lanes each; 16; 32
    y, t = W.random_points(n, big, n)
    prm = hpt.Params(tol_accept=1e-2)
    out = {}
    for p in (big, mid, small):
        st = h.new_state(p)
        st.y.copy_(torch.from_numpy(y[:p]))
        st.y_acc.copy_(st.y)
        st.tau.copy_(torch.from_numpy(np.log(0.3 + 0.7 * t[:p])))
        st.tau_acc.copy_(st.tau)
        st.dtau.fill_(0.01)
        st.accepts.fill_(1)
        st.status[5::11] = hpt.CONVERGED   # paths that are not stepped, in every warp
        h.step(st, 2, prm)
        x = torch.from_numpy(y[:p].copy()).cuda()
        h.polish(x, None, hpt.Params(polish_iters=2))
        gx = torch.from_numpy(np.conj(y[:p])).cuda()
        gx[small:] = 0   # the other solutions add zeros, in the same order
        out[p] = {f: getattr(st, f).cpu().numpy() for f in st.FIELDS}
        out[p]["x"] = x.cpu().numpy()
        out[p]["gc"] = h.adjoint(torch.from_numpy(y[:p]).cuda(), gx).cpu().numpy()[:small]
    for f, v in out[small].items():
        assert np.array_equal(v, out[big][f][:small], equal_nan=True), f
        assert np.array_equal(v, out[mid][f][:small], equal_nan=True), f
    assert (out[big]["accepts"] + out[big]["rejects"] >= 1).all()
