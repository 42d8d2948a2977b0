"""Calls captured into a CUDA graph replay to the eager results (GPU): the
step's kernels are launched as programmatic dependents of one another, and a
graph has to keep their order (small grids, which let the next kernel begin at
once, and large ones)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,p", [(0, 5, 40), (0, 14, 3000), (1, 5, 40), (1, 14, 3000), (1, 20, 200)])
@pytest.mark.parametrize("proj", [False, True], ids=["affine", "projective"])
def test_captured_steps_equal_eager(hpt, prec, n, p, proj):
    s = W.laurent_system(60 + n, n, 6, -2, 2, 8, nnz=min(n, 4))
    alpha = W.random_alpha(5, n, -1, 1)
    h = hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": alpha.tolist(), "denom": 1}, prec)
    if proj:
        h = h.homogenize()
    y, t = W.random_points(n, p, n)
    y0 = torch.from_numpy(y).cuda()
    prm = hpt.Params(tol_accept=1e-2, eps0=1e-2)
    st = h.new_state(p)

    def call():
        h.paths_init(st, y0, prm)
        h.step(st, 4, prm)

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        call()   # eager: the library's scratch is allocated here
        torch.cuda.synchronize()
        want = {f: v.clone() for f, v in st.to_host().items()}
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            call()
        for _ in range(3):
            st.y.zero_()
            st.tau.zero_()
            g.replay()
        torch.cuda.synchronize()
    for f, v in st.to_host().items():
        assert np.array_equal(v.numpy(), want[f].numpy(), equal_nan=True), f
