"""The FP64 solve at the ends of the double range (GPU): matrix entries below the
normal range keep their bits through the power-of-two equilibration, and a
pivot is refused only when the reciprocal of its square is not finite."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _directions(hpt, n, m, exps, coeffs, lifting):
    """(status, Euler direction) of one step at y = 1, t = 1, and hpt_euler_newton's
    (ok, Euler direction) there."""
    h = hpt.System(n, m, exps, coeffs, lifting, {"kind": "lower", "alpha_num": [0] * n, "denom": 1}, 0)
    st = h.new_state(1)
    st.y.fill_(1)
    st.y_acc.copy_(st.y)
    st.dtau.fill_(0.01)
    h.step(st, 1, hpt.Params(tol_accept=1e9, div_bound=1e300))
    y = torch.ones(1, n, dtype=torch.complex128).cuda()
    dE, _, ok = h.euler_newton(y, torch.zeros(1, dtype=torch.float64).cuda())
    return st.status.item(), st.dE_acc.cpu().numpy()[0], ok.item(), dE.cpu().numpy()[0]


@pytest.mark.parametrize("big,small", [(1e-300, 1e-309), (1e-307, 3e-308), (1e-305, 2e-310), (1e300, 1e290)])
def test_small_entries(hpt, big, small):
    """Rows (big, small) and (0, 1): the first unknown is 3 small / big.  Each
    of the two coefficients is rounded to its last bit twice on the way."""
    status, dE, ok, d = _directions(hpt, 2, [3, 2], [[1, 0], [0, 1], [0, 0], [0, 1], [0, 0]],
                                    [big, small, -big, 1, -1], [0, 0, 0, 3, 0])
    want = np.array([3 * (small / big), -3.0])
    ulp = 2.0 ** -52 + 2.0 ** -1074 / small
    assert status == hpt.CONVERGED and ok == 1
    for got in (dE, d):
        assert (np.abs(got - want) <= 8 * ulp * np.abs(want)).all(), got


@pytest.mark.parametrize("e,accepted", [(1e-30, True), (1e-150, True), (2e-154, True), (1e-158, False), (0.0, False)])
def test_small_pivots(hpt, e, accepted):
    """Rows (1, 0, 0), (1, e, 0), (0, 1, 1): the last pivot is e/2 after the
    equilibration, and neither rows nor columns can bring it up."""
    status, dE, ok, d = _directions(
        hpt, 3, [2, 3, 3], [[1, 0, 0], [0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 0], [0, 1, 0], [0, 0, 1], [0, 0, 0]],
        [1, -1, 1, e, -1, 1, 1, -2], [0, 0, 0, 3, 0, 0, 0, 0])
    assert (status == hpt.CONVERGED) == accepted and ok == int(accepted)
    if accepted:
        for got in (dE, d):
            assert np.abs(got - np.array([0, -3, 3])).max() <= 1e-13, got
