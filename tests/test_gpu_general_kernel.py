"""The FP64 kernels for exponents beyond the fixed point's range (GPU):
evaluation, step, directions, polish and adjoint of systems with one monomial
of sum |a_j| > 1,024 or t-exponent >= 2^31, at every size of the kernel (n <= 8,
16, 24, 32), against the oracle and against the same system just inside the
range; and a batch in which exactly one system is beyond it.

Tolerances: evaluations 1e-11 of the sum of term magnitudes (the repository's
FP64 bound); directions that times the condition of the matrix solved."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import cells

import _util

pytestmark = pytest.mark.gpu
SIZES = [1, 8, 12, 16, 20, 28, 32]


def _system(n, far):
    """far: ("sum", s) a monomial of sum |a_j| = s with a coefficient of its own;
    ("texp", e) a monomial with t-exponent e and coefficient 0."""
    s = W.laurent_system(90 + n, n, 4 if n == 1 else 6, -2, 2, 8, nnz=min(n, 4))
    i = s.m[0] - 1
    lift = s.lifting.copy()
    lift[0] = 0
    ex, co = s.exponents.copy(), s.coeffs.copy()
    if far[0] == "sum":
        a = np.zeros(n, np.int32)
        a[0] = far[1] if n == 1 else far[1] // 2
        if n > 1:
            a[n - 1] = -(far[1] - far[1] // 2)
        ex[i] = a
        assert np.abs(a).sum() == far[1]
    else:
        lift[i] = far[1]
        co[i] = 0.0
    return W.LaurentSystem(n, s.m, ex, co, lift)


def _handle(hpt, oracle_mod, s):
    h = hpt.System.from_laurent(s, {"kind": "explicit", "alpha_num": [0] * s.n, "beta_num": [0] * s.n, "denom": 1}, 0)
    te = h.texp()
    return h, oracle_mod.System(s, te["e"], te["D"])


FAR = [("sum", 1024), ("sum", 1025), ("sum", 1500), ("texp", (1 << 31) - 1), ("texp", 1 << 31)]


@pytest.mark.parametrize("far", FAR, ids=lambda f: f"{f[0]}{f[1]}")
@pytest.mark.parametrize("n", SIZES)
def test_calls_match_the_oracle(hpt, oracle_mod, n, far):
    s = _system(n, far)
    h, osys = _handle(hpt, oracle_mod, s)
    p = 67
    y, t = W.torus_points(n, p, n, 0.004)
    t = 0.3 + 0.7 * t
    tau = np.log(t)
    yd, td, taud = torch.from_numpy(y).cuda(), torch.from_numpy(t).cuda(), torch.from_numpy(tau).cuda()
    H, Hy, Ht = (a.cpu().numpy() for a in h.eval(yd, td))
    Ho, Hyo, Hto = osys.eval(y, tau)
    SH, SHy, SHt = osys.scale(y, tau)
    assert max(_util.scaled_err(H, Ho, SH), _util.scaled_err(Hy, Hyo, SHy),
               _util.scaled_err(Ht, Hto / t[:, None], SHt / t[:, None])) <= 1e-11

    def close(got, want, tau_, keep):
        """Solutions of the Jacobian at (y, tau_), each within its condition."""
        J = osys.eval(y, tau_)[1] * y[:, None, :]
        J = J / np.abs(J).max(-1, keepdims=True)
        J = J / np.abs(J).max(-2, keepdims=True)
        kappa = np.linalg.cond(J)
        assert (kappa < 1e6).sum() >= p // 2
        k = keep & (kappa < 1e6)
        err = np.abs(got[k] - want[k]).max(-1) / np.maximum(1.0, np.abs(want[k]).max(-1))
        assert (err <= 1e-11 * kappa[k]).all(), (err / kappa[k]).max()

    dE, dN, ok = (a.cpu().numpy() for a in h.euler_newton(yd, taud))
    dEo, dNo, oko = osys.directions(y, tau)
    for a, b in ((dE, dEo), (dN, dNo)):
        close(a, b, tau, (ok == 1) & oko)
    # a step that accepts the corrected point, and one polish iteration at t = 1
    st = h.new_state(p)
    st.y.copy_(yd)
    st.y_acc.copy_(yd)
    st.tau.copy_(taud)
    st.tau_acc.copy_(taud)
    st.dtau.fill_(1e-3)
    h.step(st, 1, hpt.Params(tol_accept=1e30, div_bound=1e300))
    acc = st.accepts.cpu().numpy() == 1
    assert acc.sum() >= 0.9 * p
    close(st.y_acc.cpu().numpy(), y + dNo, tau, acc & oko)
    close(st.dE_acc.cpu().numpy(), dEo, tau, acc & oko)
    x = yd.clone()
    h.polish(x, None, hpt.Params(polish_iters=1, polish_tol=1e-300))
    dN1, ok1 = osys.directions(y, 0.0)[1:]
    close(x.cpu().numpy(), y + dN1, 0.0, ok1)
    # the adjoint, solution by solution
    q = 5
    gx = np.conj(y[:q]) + 1j
    for i in range(q):
        g = h.adjoint(yd[i:i + 1], torch.from_numpy(gx[i:i + 1]).cuda()).cpu().numpy()
        go = osys.adjoint(y[i:i + 1], gx[i:i + 1])
        J = osys.eval(y[i:i + 1], 0.0)[1][0] * y[i]
        assert np.abs(g - go).max() <= 1e-11 * np.linalg.cond(J) * np.abs(go).max()


def _shape(n, seed):
    s, pairs = W.paper_shape(n, 7 * n, attempt=seed)
    return s, pairs


def test_batch_with_one_system_beyond_the_range(hpt, oracle_mod):
    """One system with a monomial of sum |a_j| = 1,100 sends the polish of every system of the batch
    through the general kernels: same statuses and steps as the batch without
    it, solutions within 1e-9; its own solutions match the oracle's."""
    a = np.array([220, -220, 220, -220, 220])   # the mixed form takes |a_j| <= 256
    ex = [a, 0 * a, np.eye(5, dtype=int)[1]]
    co, lift = [1, np.exp(0.3j), 0.01], [0, 0, 3]
    for k in range(1, 5):
        ex += [2 * np.eye(5, dtype=int)[k], 0 * a, np.eye(5, dtype=int)[k - 1]]
        co += [1, np.exp(1j * k), 0.01]
        lift += [0, 0, 2]
    far = W.LaurentSystem(5, [3] * 5, ex, co, lift)
    fp = [[0, 1]] * 5
    sizes = [6, 13, 21, 28]
    cases = [_shape(n, 0) for n in sizes]
    paths = [60, 33, 130, 40]
    ks = [np.zeros((p, s.n), np.int64) for (s, _), p in zip(cases, paths)]
    for k in ks:
        k[:, 0] = np.arange(len(k))
    y0 = [cells.start_points_at(s, pr, k) for (s, pr), k in zip(cases, ks)]
    kf = np.zeros((50, 5), np.int64)
    kf[:, 0] = np.arange(50)
    yf = cells.start_points_at(far, fp, kf)
    mk = lambda s, pr: hpt.System.from_laurent(s, {"kind": "pairs", "pairs": pr}, 1)   # noqa: E731
    hs, hf = [mk(*c) for c in cases], mk(far, fp)
    prm = hpt.Params(tol_accept=3e-3)

    def run(handles, ys):
        flat = torch.from_numpy(np.concatenate([y.reshape(-1) for y in ys])).cuda()
        b = hpt.Batch(handles)
        return [a.cpu().numpy() for a in b.track(flat, [len(y) for y in ys], prm)]

    x0, st0, sp0 = run(hs, y0)
    x1, st1, sp1 = run(hs[:2] + [hf] + hs[2:], y0[:2] + [yf] + y0[2:])
    P = sum(paths[:2])
    V = sum(p * n for p, n in zip(paths[:2], sizes[:2]))
    keep = np.r_[0:P, P + 50:len(st1)]
    assert np.array_equal(st0, st1[keep]) and np.array_equal(sp0, sp1[keep])
    xf = x1[V:V + 250].reshape(50, 5)
    xo = np.concatenate([x1[:V], x1[V + 250:]])
    vo = po = 0
    for n, p in zip(sizes, paths):
        a, b = x0[vo:vo + p * n].reshape(p, n), xo[vo:vo + p * n].reshape(p, n)
        conv = st0[po:po + p] == hpt.CONVERGED
        assert conv.sum() >= p // 4, (n, np.bincount(st0[po:po + p]))
        rel = np.abs(a[conv] - b[conv]).max(-1) / np.maximum(1.0, np.abs(a[conv]).max(-1))
        assert rel.max() < 1e-9, n
        vo += p * n
        po += p
    te = cells.t_exponents(far, {"kind": "pairs", "pairs": fp})
    xr, sto, _, _ = oracle_mod.System(far, te["e"], te["D"]).track(oracle_mod.Params(), yf, cells.tau0(te["e"], te["D"]))
    assert (sto == oracle_mod.CONVERGED).all() and (st1[P:P + 50] == hpt.CONVERGED).all()
    assert _util.match_solutions(xf, xr) < 1e-9
