"""The fixed-point FP64 evaluation on the GPU where it can go wrong: monomials
without nonzero exponents, one to 32 of them, ragged supports, t-exponents
over a denominator, zero coefficients, tiles of 1, 31, 33 points,
points without a logarithm, and the exponents that go to the general kernel.
Tolerance: the repository's 1e-11 of the sum of term magnitudes for FP64."""
import numpy as np
import pytest
import torch

import workloads as W

import _util

pytestmark = pytest.mark.gpu


def _system(n, m, lo, hi, seed, zero_coeff=False):
    rng = np.random.default_rng(seed)
    M = sum(m)
    exps = np.zeros((M, n), np.int32)
    for i in range(M):
        k = int(rng.integers(0, n + 1))   # 0..n nonzeros: constants too
        exps[i, rng.choice(n, k, replace=False)] = rng.integers(lo, hi + 1, size=k)
    c = np.exp(0.3 * rng.standard_normal(M) + 2j * np.pi * rng.random(M))
    if zero_coeff:
        c[::5] = 0.0
    lift = rng.integers(0, 20, size=M)
    return W.LaurentSystem(n, m, exps, c, lift)


def _compare(hpt, oracle_mod, s, alpha, denom, y, t, tol=1e-11):
    h = hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": alpha, "denom": denom}, 0)
    te = h.texp()
    osys = oracle_mod.System(s, te["e"], denom)
    H, Hy, Ht = (a.cpu().numpy() for a in h.eval(torch.from_numpy(y).cuda(), torch.from_numpy(t).cuda()))
    Ho, Hyo, Hto = osys.eval(y, np.log(t))
    SH, SHy, SHt = osys.scale(y, np.log(t))
    errs = (_util.scaled_err(H, Ho, SH), _util.scaled_err(Hy, Hyo, SHy), _util.scaled_err(Ht, Hto / t[:, None], SHt / t[:, None]))
    assert max(errs) <= tol, errs
    return h, H, Hy, Ht


@pytest.mark.parametrize("n,m", [(1, [3]), (3, [1, 2, 9]), (5, [2, 40, 3, 7, 130]), (17, [4] * 17), (32, [5] * 31 + [64])])
@pytest.mark.parametrize("p", [1, 33])
def test_parity(hpt, oracle_mod, n, m, p):
    s = _system(n, m, -3, 3, n)
    rng = np.random.default_rng(p)
    alpha = rng.integers(-2, 3, size=n).tolist()
    y, t = W.random_points(5, p, n)
    y = y / np.abs(y) * np.abs(y) ** 0.5
    _compare(hpt, oracle_mod, s, alpha, 3, y, 0.3 + 0.7 * t)


def test_zero_coefficients_and_wide_range(hpt, oracle_mod):
    s = _system(4, [5, 6, 7, 8], -2, 2, 9, zero_coeff=True)
    rng = np.random.default_rng(1)
    y = np.exp(30 * rng.standard_normal((31, 4)) + 2j * np.pi * rng.random((31, 4)))   # |y| to 1e+-40
    _compare(hpt, oracle_mod, s, [0] * 4, 1, y, np.full(31, 0.5))


def test_beyond_the_range_goes_to_the_general_kernel(hpt, oracle_mod):
    """sum |a_j| = 1,100 > 1,024, at points on the unit torus (1,100 factors
    and a phase of 1,100 angles: about 1e-12 in double)."""
    s = _system(3, [4, 5, 6], -2, 2, 4)
    s.exponents[2] = [600, -500, 0]
    y = W.torus_points(8, 37, 3, 0.005)[0]
    _compare(hpt, oracle_mod, s, [0] * 3, 1, y, np.full(37, 0.7))


def test_points_without_a_logarithm(hpt, oracle_mod):
    """A zero, infinite or NaN coordinate makes that point NaN in every entry
    and leaves the other points' bits alone."""
    s = _system(4, [5, 6, 7, 8], -2, 2, 9)
    y, t = W.random_points(5, 64, 4)
    t = 0.2 + 0.8 * t
    h, H0, Hy0, Ht0 = _compare(hpt, oracle_mod, s, [0] * 4, 1, y, t)
    bad = y.copy()
    bad[3, 0] = 0.0
    bad[40, 1] = np.inf
    bad[41, 2] = np.nan
    H, Hy, Ht = (a.cpu().numpy() for a in h.eval(torch.from_numpy(bad).cuda(), torch.from_numpy(t).cuda()))
    rows = np.array([3, 40, 41])
    for a, b in ((H, H0), (Hy, Hy0), (Ht, Ht0)):
        assert np.isnan(a[rows]).all()
        assert np.array_equal(np.delete(a, rows, 0), np.delete(b, rows, 0))
