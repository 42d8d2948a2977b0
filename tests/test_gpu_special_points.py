"""FP64 evaluation at coordinates 0 and infinity and at t = 0 (GPU): the values
of exp(<a, log y> + e/D log t) as written, in numpy.  A monomial with a positive
power of a zero coordinate (a negative one of an infinite one) is 0; one that
lacks the coordinate takes 0 times infinity and is NaN with its equation; every
other point keeps its bits."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _dense(s, e, denom, y, t):
    """H, H_y, H_t by the formula, with the products 0 * inf it makes."""
    with np.errstate(all="ignore"):
        p, n = y.shape
        M = s.M
        lr, li = np.log(np.abs(y)), np.angle(y)
        a = s.exponents.astype(float)
        te = np.asarray(e, float) / denom
        H, Hy, Ht = np.zeros((p, n), complex), np.zeros((p, n, n), complex), np.zeros((p, n), complex)
        tau = np.log(t)
        r2 = y.real ** 2 + y.imag ** 2
        iy = y.real / r2 - 1j * (y.imag / r2)
        row = np.repeat(np.arange(n), s.m)
        for i in range(M):
            wr, wi = te[i] * tau, np.zeros(p)
            for j in range(n):
                wr, wi = wr + a[i, j] * lr[:, j], wi + a[i, j] * li[:, j]
            m = np.exp(wr)
            E = np.where(m == 0, 0, m) * np.exp(1j * wi)
            E = np.where(np.isfinite(wr) | (wr == -np.inf), E, np.nan) * s.coeffs[i]
            E = np.where(np.isnan(wi), np.nan, E)
            H[:, row[i]] += E
            Ht[:, row[i]] += te[i] * E
            Hy[:, row[i]] += a[i] * E[:, None]
        for q, k in zip(*np.nonzero(~np.isfinite(H))):
            H[q, k] = Ht[q, k] = complex(np.nan, np.nan)
            Hy[q, k] = complex(np.nan, np.nan)
        out = np.empty_like(Hy)   # componentwise: numpy's complex product spreads a NaN as the kernel does
        out.real = Hy.real * iy.real[:, None] - Hy.imag * iy.imag[:, None]
        out.imag = Hy.real * iy.imag[:, None] + Hy.imag * iy.real[:, None]
        ht = np.empty_like(Ht)
        ht.real, ht.imag = Ht.real * (1 / t)[:, None], Ht.imag * (1 / t)[:, None]
    return H, out, ht


def _system(n, m, seed):
    """Equation k has positive powers of variable k in every monomial, others mixed."""
    rng = np.random.default_rng(seed)
    exps = rng.integers(-2, 3, size=(n * m, n))
    for k in range(n):
        exps[k * m:(k + 1) * m, k] = rng.integers(1, 4, size=m)
        if k % 3 == 2:
            exps[k * m:(k + 1) * m, k] *= -1
    c = np.exp(0.3 * rng.standard_normal(n * m) + 2j * np.pi * rng.random(n * m))
    c[1] = 0.0
    return W.LaurentSystem(n, [m] * n, exps, c, rng.integers(0, 5, size=n * m) + 1)


@pytest.mark.parametrize("n,m", [(1, 3), (2, 4), (7, 5), (20, 3)])
def test_zero_and_infinite_coordinates(hpt, n, m):
    s = _system(n, m, 10 * n)
    h = hpt.System.from_laurent(s, {"kind": "explicit", "alpha_num": [0] * n, "beta_num": [0] * n, "denom": 1}, 0)
    te = h.texp()
    rng = np.random.default_rng(n)
    p = 70
    y = np.exp(0.3 * rng.standard_normal((p, n)) + 2j * np.pi * rng.random((p, n)))
    t = rng.uniform(0.3, 1.0, p)
    for q in range(4, p, 3):
        y[q, rng.integers(0, n)] = rng.choice([0.0, np.inf])
    y[5, 0] = complex(0.5, -np.inf)
    y[9, n - 1] = np.nan
    y[11] = 0.0
    y[13, 0], y[13, n - 1] = 0.0, np.inf
    t[6::10] = 0.0
    H, Hy, Ht = (a.cpu().numpy() for a in h.eval(torch.from_numpy(y).cuda(), torch.from_numpy(t).cuda()))
    Ho, Hyo, Hto = _dense(s, te["e"], te["D"], y, t)
    for a, b in ((H, Ho), (Hy, Hyo), (Ht, Hto)):
        for x, z in ((a.real, b.real), (a.imag, b.imag)):
            assert np.array_equal(np.isfinite(x), np.isfinite(z))
            f = np.isfinite(z)
            # terms of modulus up to about (e^0.9)^(2 n), all weighted by up to 3
            assert np.abs(x[f] - z[f]).max() <= 1e-11 * max(1.0, np.abs(z[f]).max())
    assert np.isfinite(Ho[4:]).any() and (Ho[4:] == 0).any() and np.isnan(Ho).any()
    good = np.isfinite(y).all(1) & (y != 0).all(1) & (t > 0)
    only = h.eval(torch.from_numpy(y[good]).cuda(), torch.from_numpy(t[good]).cuda())
    for a, b in zip((H, Hy, Ht), only):
        assert np.array_equal(a[good], b.cpu().numpy())
