"""The work that programs have this library do, as measured cases.

Every case goes through the binding's public entry points (System.eval,
paths_init + step, homogenize, euler_newton, track, adjoint, Batch.track,
binomial_start_device) the way a path-tracking program calls them.  The
supports, liftings and cells are drawn per case (`family`), the coefficients,
start points and sample points from the seed: a program that solves one
family of systems at new parameters.

Shapes: the throughput workload (n = 16, 512 monomials, 65,536 paths), the
paper's test-system shapes (n = 14 with 184 monomials, n = 24 with 324, 10 to
1,000 paths, many consecutive steps), the adjoint workload (n = 8, 12 dense
monomials per equation, 4,096 paths) and the many-systems batch (n in 4..24).
"""
import math

import numpy as np
import torch

from paper_2111_14317_gb300 import hpt

PREC = {"fp64": hpt.HPT_FP64, "mixed": hpt.HPT_MIXED}


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the headline: Euler-Newton steps of a whole path set, mixed precision
        {"name": "step_mixed_n16_p65536", "kind": "step", "prec": "mixed", "n": 16, "mono": 512, "nnz": 4,
         "lim": 2, "p": 65536, "steps": 2, "eps0": 1e-3, "predictor": 0, "family": 1},
        # the same path set in the FP64 form
        {"name": "step_fp64_n16_p65536", "kind": "step", "prec": "fp64", "n": 16, "mono": 512, "nnz": 4,
         "lim": 2, "p": 65536, "steps": 1, "eps0": 1e-3, "predictor": 0, "family": 1},
        # many consecutive steps of few paths (the paper's protocol): launches and latency
        {"name": "step_mixed_n14_p250", "kind": "step", "prec": "mixed", "n": 14, "mono": 184, "nnz": 4,
         "lim": 2, "p": 250, "steps": 50, "eps0": 1e-10, "predictor": 0, "family": 2},
        # the paper's larger shape in the FP64 form, with the cubic predictor
        {"name": "step_fp64_n24_p1000", "kind": "step", "prec": "fp64", "n": 24, "mono": 324, "nnz": 4,
         "lim": 2, "p": 1000, "steps": 10, "eps0": 1e-10, "predictor": 1, "family": 3},
        # the projective form's step (Algorithm 3 by QR)
        {"name": "proj_mixed_n16_p65536", "kind": "proj", "prec": "mixed", "n": 16, "mono": 512, "nnz": 4,
         "lim": 2, "p": 65536, "steps": 1, "eps0": 1e-3, "predictor": 0, "family": 1},
        # Euler and Newton directions in homogeneous coordinates, dense exponents, odd count
        {"name": "dirs_fp64_n8_p4999", "kind": "dirs", "prec": "fp64", "n": 8, "mono": 96, "nnz": 8,
         "lim": 2, "p": 4999, "family": 5},
        # H, H_y and H_t of a large dense system at given points, ragged supports
        {"name": "eval_mixed_n24_p20011", "kind": "eval", "prec": "mixed", "n": 24, "mono": 1300, "nnz": 24,
         "lim": 2, "p": 20011, "family": 24},
        # the smallest calls: a small system at a few hundred points
        {"name": "eval_fp64_n4_p333", "kind": "eval", "prec": "fp64", "n": 4, "mono": 20, "nnz": 4,
         "lim": 2, "p": 333, "family": 4},
        # whole tracks of one system, mixed form with the FP64 polish
        {"name": "track_mixed_n8_p4096", "kind": "track", "prec": "mixed", "n": 8, "mono": 96, "nnz": 8,
         "lim": 2, "p": 4096, "family": 5},
        # whole tracks of many systems of different sizes
        {"name": "batch_16x256", "kind": "batch", "systems": 16, "nlo": 4, "nhi": 24, "p": 256, "family": 40},
        # the backward pass: coefficient gradients at a set of solutions
        {"name": "adjoint_n8_p4096", "kind": "adjoint", "prec": "fp64", "n": 8, "mono": 96, "nnz": 8,
         "lim": 2, "p": 4096, "family": 5},
        # the start points of a cell of the paper's larger shape
        {"name": "starts_n24_p1048576", "kind": "starts", "n": 24, "mono": 324, "nnz": 4, "lim": 2,
         "p": 1 << 20, "family": 3},
    ]


def _logint(rng, lo, hi):
    return int(min(hi, max(lo, math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    """One more case of the same kinds: sizes spread over their whole ranges."""
    kind = rng.choice(["step", "step", "step", "proj", "dirs", "eval", "eval", "track", "batch", "adjoint", "starts"])
    fam = rng.randrange(1000, 1 << 20)
    if kind == "batch":
        nlo = rng.randint(2, 12)
        return {"kind": kind, "systems": rng.randint(2, 16), "nlo": nlo, "nhi": rng.randint(nlo, 24),
                "p": _logint(rng, 3, 256), "family": fam}
    if kind == "starts":
        n = rng.randint(12, 24)
        return {"kind": kind, "n": n, "mono": n * rng.randint(6, 16), "nnz": 4, "lim": 2,
                "p": _logint(rng, 100, 1 << 20), "family": fam}
    prec = rng.choice(["mixed", "fp64"])
    if kind == "track":
        n = rng.randint(2, 8)
        return {"kind": kind, "prec": prec, "n": n, "mono": n * rng.randint(4, 12), "nnz": n, "lim": 2,
                "p": _logint(rng, 8, 4096 if prec == "mixed" else 1024), "family": fam}
    if kind == "adjoint":
        n = _logint(rng, 2, 24)
        return {"kind": kind, "prec": prec, "n": n, "mono": n * rng.randint(5, 14), "nnz": min(n, rng.choice([4, 8])),
                "lim": 2, "p": _logint(rng, 10, max(10, 4096 * 8 // n)), "family": fam}
    n = _logint(rng, 2, 31 if kind in ("proj", "dirs") else 32)
    per = rng.randint(5, min(36, max(8, 2 * n)))
    nnz = rng.choice([min(4, n), n])
    c = {"kind": kind, "prec": prec, "n": n, "mono": n * per + rng.randrange(n), "nnz": nnz, "lim": 2}
    # at most the points of the largest listed case, and its work
    cap = max(64, min(65536, int(65536 * 512 * 16 / (c["mono"] * (n + nnz) * (1 if prec == "mixed" else 2)))))
    if kind in ("step", "proj"):
        c["p"] = _logint(rng, 10, cap)
        c["steps"] = max(1, min(40, cap // (2 * c["p"])))
        c["eps0"] = rng.choice([1e-10, 1e-6])
        c["predictor"] = rng.choice([0, 0, 1])
    else:
        c["p"] = _logint(rng, 10, min(cap, 40000))
    c["family"] = fam
    return c


# ---------------------------------------------------------------- inputs
def _split(n, mono):
    """Support sizes: `mono` monomials over n equations, ragged by one."""
    return [mono // n + (1 if k < mono % n else 0) for k in range(n)]


def _rows(rng, count, n, nnz, lim):
    """`count` distinct exponent vectors with at most nnz nonzeros in [-lim, lim]."""
    got, seen = [], set()
    while len(got) < count:
        if nnz >= n:
            block = rng.integers(-lim, lim + 1, size=(2 * count, n))
        else:
            block = np.zeros((2 * count, n), np.int64)
            at = np.argsort(rng.random((2 * count, n)), axis=1)[:, :nnz]
            v = rng.integers(1, lim + 1, size=(2 * count, nnz)) * rng.choice([-1, 1], size=(2 * count, nnz))
            np.put_along_axis(block, at, v, axis=1)
        for row in block:
            key = row.tobytes()
            if key not in seen and len(got) < count:
                seen.add(key)
                got.append(row)
    return np.array(got, np.int32)


def _support(n, m, nnz, lim, family, lift_hi=16):
    """Exponents, lifting and pairs of a planted cell (lifting 0 on one pair of
    every support, 1..lift_hi elsewhere) with a regular pair matrix."""
    for attempt in range(200):
        rng = np.random.default_rng([family, n, sum(m), attempt])
        exps = [_rows(rng, mk, n, nnz, lim) for mk in m]
        pairs = np.array([np.sort(rng.choice(mk, size=2, replace=False)) for mk in m], np.int32)
        V = np.array([e[b] - e[a] for e, (a, b) in zip(exps, pairs)], np.float64)
        sign, logdet = np.linalg.slogdet(V)
        if sign == 0 or logdet < 0.1 or np.linalg.cond(V) > 1e4:
            continue
        lift = []
        for mk, pr in zip(m, pairs):
            w = rng.integers(1, lift_hi + 1, size=mk)
            w[pr] = 0
            lift.append(w)
        return np.concatenate(exps), np.concatenate(lift).astype(np.int64), pairs
    raise RuntimeError("no regular cell")


def _coeffs(rng, M):
    return np.exp(2j * np.pi * rng.random(M))


def _start_points(rng, m, exps, coeffs, pairs, p):
    """p start points exp(V^-1 (log b + 2 pi i k)) of the cell, random k."""
    off = np.concatenate([[0], np.cumsum(m)[:-1]])
    a, b = off + pairs[:, 0], off + pairs[:, 1]
    V = (exps[b] - exps[a]).astype(np.float64)
    lb = np.log(-coeffs[a] / coeffs[b])
    k = rng.integers(-(1 << 20), 1 << 20, size=(p, len(m)))
    z = np.linalg.solve(V, (lb[None, :] + 2j * np.pi * k).T).T
    return np.ascontiguousarray(np.exp(z.real) * np.exp(1j * z.imag))


def _points(rng, p, n):
    """Random points: |y_j| log-normal, any phase; t in (0, 1)."""
    y = np.exp(0.5 * rng.standard_normal((p, n)) + 2j * np.pi * rng.random((p, n)))
    return y, rng.uniform(0.02, 1.0, size=p)


def _batch_shapes(case):
    """(n, support sizes) of every system of a batch: n in [nlo, nhi], supports in [n+1, min(4n, 64)]."""
    rng = np.random.default_rng([case["family"], case["systems"]])
    shapes = []
    for _ in range(case["systems"]):
        n = int(rng.integers(case["nlo"], case["nhi"] + 1))
        shapes.append((n, [int(v) for v in rng.integers(n + 1, min(4 * n, 64) + 1, size=n)]))
    return shapes


def _problem(case, seed):
    """Supports, coefficients and the seed's generator of a one-system case."""
    n, m = case["n"], _split(case["n"], case["mono"])
    exps, lift, pairs = _support(n, m, case["nnz"], case["lim"], case["family"])
    rng = np.random.default_rng([case["family"], seed])
    return n, m, exps, lift, pairs, _coeffs(rng, len(exps)), rng


def _params(case):
    kw = {"eps0": case.get("eps0", 1e-10), "predictor": case.get("predictor", 0)}
    if case.get("prec", "mixed") == "mixed":
        # the mixed form's tolerance; the cubic predictor wants a tighter one
        kw["tol_accept"] = 1e-3 if kw["predictor"] else 3e-3
    return hpt.Params(**kw)


def _system(n, m, exps, coeffs, lift, pairs, prec):
    return hpt.System(n, m, exps, coeffs, lift, {"kind": "pairs", "pairs": pairs}, PREC[prec])


def _homogeneous(rng, p, nv):
    y = np.exp(0.3 * rng.standard_normal((p, nv)) + 2j * np.pi * rng.random((p, nv)))
    return y / np.linalg.norm(y, axis=1, keepdims=True)


def _inputs(case, seed):
    """The host arrays of a one-system case: dict."""
    n, m, exps, lift, pairs, coeffs, rng = _problem(case, seed)
    d = {"n": n, "m": m, "exps": exps, "lift": lift, "pairs": pairs, "coeffs": coeffs}
    kind, p = case["kind"], case["p"]
    if kind in ("step", "proj", "track"):
        d["y"] = _start_points(rng, m, exps, coeffs, pairs, p)
    elif kind == "dirs":
        d["y"] = _homogeneous(rng, p, n + 1)
        d["tau"] = -rng.uniform(0.0, 2.0, size=p)
    elif kind == "eval":
        d["y"], d["t"] = _points(rng, p, n)
    elif kind == "adjoint":
        d["y"], _ = _points(rng, p, n)
        d["gx"] = rng.standard_normal((p, n)) + 1j * rng.standard_normal((p, n))
    return d


def _first_det(case):
    """|det V| of a case's cell, exactly (fraction-free elimination)."""
    m = _split(case["n"], case["mono"])
    exps, _, pairs = _support(case["n"], m, case["nnz"], case["lim"], case["family"])
    return abs(_adjugate(_pair_matrix(m, exps, pairs))[0])


# ---------------------------------------------------------------- a program's state and one pass
def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    d = _inputs(case, seed)
    kind = case["kind"]
    state = {"kind": kind, "case": case}
    if kind == "starts":
        # the whole enumeration or its first p points
        state["args"] = (d["n"], d["m"], d["exps"], d["coeffs"], d["pairs"])
        state["count"] = min(case["p"], _first_det(case))
        return state
    sysh = _system(d["n"], d["m"], d["exps"], d["coeffs"], d["lift"], d["pairs"], case["prec"])
    if kind in ("proj", "dirs"):
        sysh = sysh.homogenize()
    state["sys"] = sysh
    y = torch.from_numpy(d["y"]).cuda()
    if kind in ("step", "proj"):
        state["prm"] = _params(case)
        state["y0"] = y
        state["paths"] = sysh.new_state(case["p"], hermite=case["predictor"] == 1)
    elif kind == "track":
        state["prm"] = _params(case)
        state["y0"] = y
    elif kind == "dirs":
        state["y"] = y.to(sysh.cdtype)
        state["tau"] = torch.from_numpy(d["tau"]).cuda()
    elif kind == "eval":
        state["y"] = y.to(sysh.cdtype)
        state["t"] = torch.from_numpy(d["t"]).cuda()
    elif kind == "adjoint":
        state["y"] = y
        state["gx"] = torch.from_numpy(d["gx"]).cuda()
    return state


def _prepare_batch(case, seed):
    rng = np.random.default_rng([case["family"], seed])
    systems, y0 = [], []
    for i, (n, m) in enumerate(_batch_shapes(case)):
        exps, lift, pairs = _support(n, m, n, 3, case["family"] + i)
        coeffs = _coeffs(rng, len(exps))
        systems.append(_system(n, m, exps, coeffs, lift, pairs, "mixed"))
        y0.append(_start_points(rng, m, exps, coeffs, pairs, case["p"]).reshape(-1))
    return {"kind": "batch", "case": case, "batch": hpt.Batch(systems), "prm": hpt.Params(tol_accept=3e-3),
            "y0": torch.from_numpy(np.concatenate(y0)).cuda(), "paths": [case["p"]] * len(systems)}


def run(state):
    kind = state["kind"]
    if kind in ("step", "proj"):
        # start the paths and take the case's number of Euler-Newton steps
        st = state["sys"].paths_init(state["paths"], state["y0"], state["prm"])
        state["sys"].step(st, state["case"]["steps"], state["prm"])
        return {f: getattr(st, f) for f in st.FIELDS}
    if kind == "dirs":
        dE, dN, ok = state["sys"].euler_newton(state["y"], state["tau"])
        return {"dE": dE, "dN": dN, "ok": ok}
    if kind == "eval":
        H, Hy, Ht = state["sys"].eval(state["y"], state["t"])
        return {"H": H, "Hy": Hy, "Ht": Ht}
    if kind == "track":
        x, status, steps = state["sys"].track(state["y0"], state["prm"])
        return {"x": x, "status": status, "steps": steps}
    if kind == "batch":
        x, status, steps = state["batch"].track(state["y0"], state["paths"], state["prm"])
        return {"x": x, "status": status, "steps": steps}
    if kind == "adjoint":
        return {"gc": state["sys"].adjoint(state["y"], state["gx"])}
    y0, total = hpt.binomial_start_device(*state["args"], count=state["count"])
    return {"y0": y0, "total": total}


# ---------------------------------------------------------------- what a pass cannot do without
def _eval_flops(n, nv, M):
    """One point: W = z A (real and imaginary), exp of M monomials (20 each), J = E B^T."""
    return 2 * (2 * nv + 1) * M + 20 * M + 8 * (nv + 2) * M


def _solve_flops(n):
    return 8 * n ** 3 / 3 + 16 * n * n


def work(case):
    kind = case["kind"]
    if kind == "batch":
        fl = by = 0.0
        for n, m in _batch_shapes(case):
            # about 150 steps a path, then a few FP64 Newton iterations
            fl += 150.0 * case["p"] * (_eval_flops(n, n, sum(m)) + _solve_flops(n))
            by += case["p"] * (2 * n * 16 + 8)
        return {"bytes": by, "flops": fl}
    n, M, p = case["n"], case["mono"], case["p"]
    if kind == "starts":
        return {"bytes": 16.0 * n * p, "flops": 2.0 * n * p * 20}
    c = 16 if case["prec"] == "fp64" else 8
    nv = n + 1 if kind in ("proj", "dirs") else n
    per = _eval_flops(n, nv, M) + _solve_flops(nv)
    if kind in ("step", "proj"):
        arrays = 5 if case["predictor"] else 3
        state = arrays * nv * c + (4 if case["predictor"] else 3) * 8 + (6 if case["predictor"] else 5) * 4
        return {"bytes": float(p * (16 * n + state)), "flops": float(p * case["steps"] * per)}
    if kind == "track":
        return {"bytes": float(p * (2 * 16 * n + 8)), "flops": 150.0 * p * per}
    if kind == "dirs":
        return {"bytes": float(p * (3 * nv * c + 12)), "flops": float(p * per)}
    if kind == "eval":
        return {"bytes": float(p * (n * c + 8 + (n * n + 2 * n) * c)), "flops": float(p * _eval_flops(n, n, M))}
    return {"bytes": float(p * 2 * 16 * n + 16 * M), "flops": float(p * (per + 8 * M))}   # adjoint


# ---------------------------------------------------------------- the same in 64 bits, without the library
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Plain:
    """H, D_z H (z = log y) and H_tau in complex128 by the formulas: exponents
    A (M x nv), t-exponents s (M), coefficients c grouped by equation."""

    def __init__(self, m, A, s, c):
        dev = _dev()
        self.A = torch.from_numpy(np.asarray(A, np.float64)).to(dev)
        self.s = torch.from_numpy(np.asarray(s, np.float64)).to(dev)
        self.c = torch.from_numpy(np.asarray(c, np.complex128)).to(dev)
        self.off = np.concatenate([[0], np.cumsum(m)]).tolist()
        self.nv = self.A.shape[1]

    def terms(self, y, tau):
        z = torch.log(y)
        w = torch.complex(z.real @ self.A.T + tau[:, None] * self.s[None, :], z.imag @ self.A.T)
        return torch.exp(w) * self.c

    def jac(self, y, tau):
        T = self.terms(y, tau)
        n = len(self.off) - 1
        J = torch.empty(y.shape[0], n, self.nv, dtype=torch.complex128, device=y.device)
        Ht = torch.empty(y.shape[0], n, dtype=torch.complex128, device=y.device)
        H = torch.empty_like(Ht)
        for k in range(n):
            a, b = self.off[k], self.off[k + 1]
            J[:, k] = T[:, a:b] @ self.A[a:b].to(torch.complex128)
            Ht[:, k] = T[:, a:b] @ self.s[a:b].to(torch.complex128)
            H[:, k] = T[:, a:b].sum(1)
        return H, J, Ht


def _chunks(p, size=8192):
    return [slice(i, min(p, i + size)) for i in range(0, p, size)]


def _plain(d, homogeneous=False):
    """The planted cell has inner normal 0, so the t-exponents are the lifting."""
    A = d["exps"]
    if homogeneous:
        deg = A.sum(1)
        off = np.concatenate([[0], np.cumsum(d["m"])])
        top = np.concatenate([np.full(mk, deg[a:b].max()) for mk, a, b in zip(d["m"], off[:-1], off[1:])])
        A = np.concatenate([A, (top - deg)[:, None]], axis=1)
    return _Plain(d["m"], A, d["lift"], d["coeffs"])


def _directions(P, y, tau, proj):
    """(dE, dN) at the points: D_z H w = rhs, d = y w; in the projective form
    with the row y^* d = 0."""
    dE, dN = torch.empty_like(y), torch.empty_like(y)
    for q in _chunks(y.shape[0]):
        H, J, Ht = P.jac(y[q], tau[q])
        R = torch.stack([-Ht, -H], dim=2)
        if proj:
            J = torch.cat([J, (y[q].abs() ** 2).to(torch.complex128)[:, None, :]], dim=1)
            R = torch.cat([R, torch.zeros_like(R[:, :1])], dim=1)
        # rows and columns scaled to unit size: a plain elimination then loses nothing to their ranges
        r = 1.0 / J.abs().amax(2, keepdim=True).clamp_min(1e-300)
        J, R = J * r, R * r
        k = 1.0 / J.abs().amax(1, keepdim=True).clamp_min(1e-300)
        w = torch.linalg.solve(J * k, R) * k.transpose(1, 2)
        dE[q], dN[q] = y[q] * w[:, :, 0], y[q] * w[:, :, 1]
    return dE, dN


def _steps64(P, y0, tau0, prm, nsteps, proj):
    """The path state after nsteps of the step rule (include/hpt.h), as a dict
    of float tensors; whole-valued fields are kept for the rule only."""
    dev = _dev()
    p = y0.shape[0]
    if proj:
        y0 = torch.cat([y0, torch.ones(p, 1, dtype=y0.dtype, device=dev)], dim=1)
        y0 = y0 / torch.linalg.vector_norm(y0, dim=1, keepdim=True)
    f8 = {"dtype": torch.float64, "device": dev}
    s = {"y": y0.clone(), "y_acc": y0.clone(), "dE_acc": torch.zeros_like(y0), "tau": torch.full((p,), tau0, **f8),
         "tau_acc": torch.full((p,), tau0, **f8), "dtau": torch.full((p,), prm.dtau_init, **f8),
         "y_prev": torch.zeros_like(y0), "dE_prev": torch.zeros_like(y0), "tau_prev": torch.full((p,), tau0, **f8)}
    i8 = {"dtype": torch.int64, "device": dev}
    status, steps, accepts, streak = (torch.zeros(p, **i8) for _ in range(4))
    herm = torch.zeros(p, dtype=torch.bool, device=dev)

    def pick(mask, a, b):
        return torch.where(mask[:, None] if a.dim() == 2 else mask, a, b)

    for _ in range(nsteps):
        act = torch.nonzero(status == 0).squeeze(1)
        if act.numel() == 0:
            break
        v = {k: t[act] for k, t in s.items()}
        st, ac, sk, hm = status[act], accepts[act], streak[act], herm[act]
        sp = steps[act] + 1
        dE, dN = _directions(P, v["y"], v["tau"], proj)
        bad = ~(torch.isfinite(dE.abs().sum(1)) & torch.isfinite(dN.abs().sum(1)))
        err = dN.abs().amax(1) / v["y"].abs().amax(1).clamp_min(1.0)
        ok = ~bad & (err <= prm.tol_accept)
        new = v["y"] + dN
        inv = 1.0 / torch.linalg.vector_norm(new, dim=1, keepdim=True) if proj else torch.ones(len(act), 1, **f8)
        new, dEn = new * inv, dE * inv
        keep = ok & (ac >= 1) if prm.predictor == 1 else torch.zeros_like(ok)
        for prev, cur in (("y_prev", "y_acc"), ("dE_prev", "dE_acc"), ("tau_prev", "tau_acc")):
            v[prev] = pick(keep, v[cur], v[prev])
        v["y_acc"], v["dE_acc"] = pick(ok, new, v["y_acc"]), pick(ok, dEn, v["dE_acc"])
        v["tau_acc"] = pick(ok, v["tau"], v["tau_acc"])
        ac, sk = ac + ok, torch.where(ok, sk + 1, torch.zeros_like(sk))
        size = new[:, :-1].abs() / new[:, -1:].abs() if proj else new.abs()
        div = ok & ((size >= prm.div_bound) | (size <= 1.0 / prm.div_bound)).any(1)
        end = ok & (v["tau_acc"] == 0)
        div, end = (div, end & ~div) if proj else (div & ~end, end)
        st = torch.where(div, torch.full_like(st, 2), torch.where(end, torch.ones_like(st), st))
        grow = ok & ~div & ~end & (sk >= prm.grow_after)
        v["dtau"] = pick(grow, (v["dtau"] * prm.grow).clamp_max(prm.dtau_max), v["dtau"])
        sk = torch.where(grow, torch.zeros_like(sk), sk)
        first = ~ok & (ac == 0)
        st = torch.where(first & bad, torch.full_like(st, 4), st)
        fix = first & ~bad
        v["y"], v["y_acc"] = pick(fix, new, v["y"]), pick(fix, new, v["y_acc"])
        retry = ~ok & ~first & hm
        shrink = ~ok & ~first & ~hm
        v["dtau"] = pick(shrink, v["dtau"] * prm.shrink, v["dtau"])
        under = shrink & (v["dtau"] < prm.dtau_min)
        st = torch.where(under, torch.full_like(st, 3), st)
        pred = ~(div | end | first | under)
        h = torch.minimum(v["dtau"], -v["tau_acc"])
        d = v["tau_acc"] - v["tau_prev"]
        cubic = pred & ~retry & (ac >= 2) & (d > 0) if prm.predictor == 1 else torch.zeros_like(ok)
        plain = v["y_acc"] + h[:, None] * v["dE_acc"]
        u = (1.0 + h / torch.where(d > 0, d, torch.ones_like(d)))[:, None]
        ph = torch.ones(len(act), 1, dtype=torch.complex128, device=dev)
        if proj:
            dot = (v["y_acc"].conj() * v["y_prev"]).sum(1, keepdim=True)
            ph = torch.where(dot.abs() > 0, dot.conj() / dot.abs().clamp_min(1e-300), ph)
        curve = ((2 * u ** 3 - 3 * u ** 2 + 1) * (v["y_prev"] * ph) + (u ** 3 - 2 * u ** 2 + u) * d[:, None] * (v["dE_prev"] * ph)
                 + (3 * u ** 2 - 2 * u ** 3) * v["y_acc"] + (u ** 3 - u ** 2) * d[:, None] * v["dE_acc"])
        v["y"] = pick(pred, pick(cubic, curve, plain), v["y"])
        v["tau"] = pick(pred, v["tau_acc"] + h, v["tau"])
        st = torch.where((pred | fix) & (sp >= prm.max_steps), torch.full_like(st, 5), st)
        if prm.predictor == 1:
            herm[act] = torch.where(pred, cubic, hm)
        for k in s:
            s[k][act] = v[k]
        status[act], accepts[act], streak[act], steps[act] = st, ac, sk, sp
    return s, status


def _polish64(P, x, converged):
    """Newton at t = 1 of the converged rows to rounding."""
    x = x.clone()
    if converged.any():
        v = x[converged]
        zero = torch.zeros(v.shape[0], dtype=torch.float64, device=v.device)
        for _ in range(6):
            v = v + _directions(P, v, zero, False)[1]
        x[converged] = v
    return x


def _tau0(lift, eps0):
    return math.log(eps0) / float(lift[lift > 0].min())


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None   # tens of systems through hundreds of steps each
    d = _inputs(case, seed)
    if kind == "starts":
        return _exact_starts(case, d)
    dev = _dev()
    y = torch.from_numpy(d["y"]).to(dev)
    P = _plain(d, kind in ("proj", "dirs"))
    if case["prec"] == "mixed" and kind not in ("track", "adjoint", "step", "proj"):
        y = y.to(torch.complex64).to(torch.complex128)   # the inputs that the form takes
    if kind in ("step", "proj"):
        prm = _params(case)
        s, _ = _steps64(P, y, _tau0(d["lift"], prm.eps0), prm, case["steps"], kind == "proj")
        whole = ("status", "steps", "accepts", "rejects", "streak", "hermite")
        names = hpt.PathState.BASE + (hpt.PathState.PREV if case["predictor"] else ())
        return {f: None if f in whole else s[f] for f in names}
    if kind == "track":
        prm = _params(case)
        s, status = _steps64(P, y, _tau0(d["lift"], prm.eps0), prm, 2000, False)
        return {"x": _polish64(P, s["y_acc"], status == 1), "status": None, "steps": None}
    if kind == "dirs":
        dE, dN = _directions(P, y, torch.from_numpy(d["tau"]).to(dev), True)
        return {"dE": dE, "dN": dN, "ok": None}
    if kind == "eval":
        t = torch.from_numpy(d["t"]).to(dev)
        parts = []
        for q in _chunks(y.shape[0]):
            H, J, Ht = P.jac(y[q], torch.log(t[q]))
            parts.append((H, J / y[q][:, None, :], Ht / t[q][:, None]))
        H, Hy, Ht = (torch.cat(v) for v in zip(*parts))
        return {"H": H, "Hy": Hy, "Ht": Ht}
    gx = torch.from_numpy(d["gx"]).to(dev)
    gc = torch.zeros(len(d["exps"]), dtype=torch.complex128, device=dev)
    zero = torch.zeros(y.shape[0], dtype=torch.float64, device=dev)
    for q in _chunks(y.shape[0]):
        _, J, _ = P.jac(y[q], zero[q])
        J = J / y[q][:, None, :]
        lam = torch.linalg.solve(J.conj().transpose(1, 2), gx[q])
        x = P.terms(y[q], zero[q]) / P.c
        eq = torch.from_numpy(np.repeat(np.arange(d["n"]), d["m"])).to(dev)
        gc -= (lam[:, eq] * x.conj()).sum(0)
    return {"gc": gc}


# ---- start points: integer bookkeeping of a cell in Python integers
def _pair_matrix(m, exps, pairs):
    off = np.concatenate([[0], np.cumsum(m)[:-1]])
    return [[int(v) for v in exps[o + b] - exps[o + a]] for o, (a, b) in zip(off, pairs)]


def _adjugate(V):
    """(det V, adj V) of an integer matrix, by fraction-free elimination of [V | I]."""
    n = len(V)
    A = [list(r) + [1 if i == j else 0 for j in range(n)] for i, r in enumerate(V)]
    prev, sign = 1, 1
    for c in range(n):
        piv = next((r for r in range(c, n) if A[r][c]), None)
        if piv is None:
            return 0, None
        if piv != c:
            A[c], A[piv] = A[piv], A[c]
            sign = -sign
        for r in range(n):
            if r != c:
                f = A[r][c]
                A[r] = [(A[c][c] * a - f * b) // prev for a, b in zip(A[r], A[c])]
        prev = A[c][c]
    # every row now reads prev x_r = right-hand side, prev = sign * det V
    return sign * prev, [[sign * v for v in A[r][n:]] for r in range(n)]


def _lattice_diagonal(V, D):
    """The diagonal of the triangular basis of the lattice V Z^n, rows from the last."""
    n = len(V)
    H = [[v % D for v in row] for row in V]
    R, h = D, [1] * n
    for i in range(n - 1, -1, -1):
        for j in range(i):
            while H[i][j]:
                q = H[i][i] // H[i][j]
                for r in range(i + 1):
                    H[r][i], H[r][j] = H[r][j], (H[r][i] - q * H[r][j]) % R
        g = math.gcd(H[i][i], R)
        h[i] = g
        R //= g
        if R == 1:
            break
        u = pow((H[i][i] // g) % R, -1, R) if math.gcd(H[i][i] // g, R) == 1 else None
        if u is None:   # the pivot's cofactor shares a factor with the modulus: not reduced further here
            return None
        for r in range(i):
            for j in range(i):
                H[r][j] %= R
    return h


def _exact_starts(case, d):
    V = _pair_matrix(d["m"], d["exps"], d["pairs"])
    det, adj = _adjugate(V)
    D = abs(det)
    h = _lattice_diagonal(V, D)
    count = min(case["p"], D)
    if h is None or math.prod(h) != D:
        return None
    n = case["n"]
    off = np.concatenate([[0], np.cumsum(d["m"])[:-1]])
    lb = np.log(-d["coeffs"][off + d["pairs"][:, 0]] / d["coeffs"][off + d["pairs"][:, 1]])
    z0 = np.linalg.solve(np.array(V, np.float64), lb)
    out = np.empty((count, n), np.complex128)
    sgn = 1 if det > 0 else -1
    for r in range(n):
        # numerators sum_j adj_rj k_j mod D over the mixed radix of k, last digit fastest
        num = np.zeros(1, np.uint64)
        for j in range(n - 1, -1, -1):
            base, want = num, min(count, len(num) * h[j])
            a, digit = (sgn * adj[r][j]) % D, 1
            while len(num) < want:   # digits [0, digit) done: append [digit, 2 digit)
                step = np.uint64((a * digit) % D)
                num = np.concatenate([num, (num + step) % np.uint64(D)])[:want]
                digit *= 2
            num = num[:want]
            if len(base) >= count:
                break
        ang = z0[r].imag + 2.0 * np.pi * (num.astype(np.float64) / float(D))
        out[:, r] = np.exp(z0[r].real) * (np.cos(ang) + 1j * np.sin(ang))
    return {"y0": out, "total": None}
