"""Measured cases of the interior-point conic solver.

Every case is one call sequence of a program that uses the solver, through the
Python binding: the solver object exists (its host analysis done, its buffers on
the GPU), new data may arrive as host arrays, and the answer is read back as host
arrays.  Problem families and sizes are those of ``workloads.py``, the tests and
``bench.py``.

Settings: the library's defaults for the factor precision, with the termination
tolerance 1e-6 (one of the two the method is evaluated at) where a case runs to
its end.  A case with ``iters`` is a solve on an iteration budget
(``max_iter``), as a real-time loop runs it; it keeps the iterates well inside
the cones, where two correct implementations agree to many digits (at the end of
a solve of a degenerate problem the multipliers are not unique).
"""
import math

import numpy as np
import torch

from paper_2412_19027_gb300 import clr, workloads as W

EPS = 1e-6


def listed():
    return [
        # one dense KKT system inside a control period or a captured graph, device pointers in and out
        {"name": "dense_kkt_n48", "kind": "dense_kkt", "n": 48},
        # the small QP (n = 50, m = 100), solved to the default 1e-8: launches and latency
        {"name": "qp_n50_fp64", "kind": "qp", "n": 50, "bits": 64},
        # one model-predictive controller: a new state arrives, the plan is solved again
        {"name": "mpc_one_fp64", "kind": "mpc", "T": 20, "nx": 8, "nu": 3, "count": 1, "bits": 64},
        # 64 controllers of uneven horizon and size in one cohort, each with its new state
        {"name": "mpc_cohort64_fp64", "kind": "mpc", "T": 0, "nx": 0, "nu": 0, "count": 64, "bits": 64},
        # mixed-cone QP (nonneg, SOC, exp, pow rows; dense P) at the benchmark's size, FP64 factor
        {"name": "mixed_n2000_fp64", "kind": "mixed", "n": 2000, "iters": 6, "bits": 64},
        # entropy maximisation, one exponential cone per variable
        {"name": "entropy_n600_fp64", "kind": "entropy", "n": 600, "iters": 5, "bits": 64},
        # portfolio re-optimisation with new expected returns, the smallest of the published sizes, FP32 factor
        {"name": "portfolio_n5000_fp32", "kind": "portfolio", "n": 5000, "bits": 32},
        # robust regression with the Huber loss, FP64 factor
        {"name": "huber_n1000_fp64", "kind": "huber", "n": 1000, "bits": 64},
        # small SDP with cones of mixed orders 2 .. 16, FP64 factor
        {"name": "psd_mixed_fp64", "kind": "psd_mixed", "per_order": 2, "iters": 4, "bits": 64},
        # batch of PSD(10) cones (a fifth of the benchmark's), FP32 factor
        {"name": "psd_batch_n4000_fp32", "kind": "psd_batch", "n": 4000, "order": 10, "iters": 3, "bits": 32},
        # large sparse LP/QP with a banded matrix: the first iterations of a long solve, both factors
        {"name": "banded_n20000_fp64", "kind": "banded", "n": 20000, "iters": 4, "bits": 64},
        {"name": "banded_n40000_fp32", "kind": "banded", "n": 40000, "iters": 3, "bits": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense_kkt", "qp", "mpc", "mpc", "mixed", "entropy", "portfolio", "huber", "psd_mixed",
                       "psd_batch", "banded", "banded"])
    bits = rng.choice([32, 64])
    if kind == "dense_kkt":
        return {"kind": kind, "n": _log_int(rng, 4, 128)}
    if kind == "qp":
        return {"kind": kind, "n": _log_int(rng, 10, 200), "bits": 64}
    if kind == "mpc":
        if rng.random() < 0.5:
            return {"kind": kind, "T": rng.randint(10, 50), "nx": rng.randint(4, 12), "nu": rng.randint(2, 4),
                    "count": 1, "bits": 64}
        return {"kind": kind, "T": 0, "nx": 0, "nu": 0, "count": _log_int(rng, 5, 100), "bits": 64}
    if kind == "mixed":
        return {"kind": kind, "n": _log_int(rng, 200, 2000), "iters": rng.randint(4, 6), "bits": 64}
    if kind == "entropy":
        return {"kind": kind, "n": _log_int(rng, 50, 600), "iters": rng.randint(3, 5), "bits": 64}
    if kind == "portfolio":
        return {"kind": kind, "n": _log_int(rng, 400, 4800), "bits": bits}
    if kind == "huber":
        return {"kind": kind, "n": _log_int(rng, 150, 1200), "bits": bits}
    if kind == "psd_mixed":
        return {"kind": kind, "per_order": rng.randint(1, 6), "iters": rng.randint(3, 4), "bits": 64}
    if kind == "psd_batch":
        return {"kind": kind, "n": 10 * _log_int(rng, 60, 350), "order": rng.randint(5, 12), "iters": 3, "bits": bits}
    return {"kind": kind, "n": _log_int(rng, 1500, 36000 if bits == 32 else 18000), "iters": rng.randint(2, 3),
            "bits": bits}


# ---------------------------------------------------------------- problems
def _problem(case, seed):
    k = case["kind"]
    if k == "qp":  # a unique, nondegenerate optimum: n active rows, n inactive ones
        n = case["n"]
        return W.unique_qp(seed, n=n, n_eq=n // 5, n_inactive=n, rank=5)
    if k == "mixed":  # the benchmark's proportions; inequalities in the place of its equations, some of which are empty
        n = case["n"]
        return W.mixed_cone(seed, n=n, n_zero=0, n_nonneg=7 * n // 4, n_soc=n // 4, n_exp=n // 20, n_pow=n // 20)
    if k == "entropy":
        return W.entropy_max(seed, n=case["n"])
    if k == "portfolio":
        return W.portfolio_qp(seed, n=case["n"])
    if k == "huber":
        return W.huber_qp(seed, n=case["n"])
    if k == "psd_mixed":
        return W.psd_mixed(seed, n=30 * case["per_order"], per_order=case["per_order"],
                           n_nonneg=10 * case["per_order"])
    if k == "psd_batch":  # a tenth as many cones as variables, a quarter as many nonnegative rows
        n = case["n"]
        return W.psd_batch(seed, n=n, n_psd=n // 10, psd_k=case["order"], n_nonneg=n // 4)
    if k == "banded":  # inequality rows only: with the first quarter as equations these are rank deficient
        return W.banded_lp(seed, n=case["n"], n_zero=0)
    raise ValueError(k)


def _mpc_pairs(case, seed):
    """(problem as set up, the same with a later state) of each controller."""
    out = []
    for i in range(case["count"]):
        sd = 1000 * seed + i
        size = {"T": case["T"] or 10 + 17 * i % 41, "nx": case["nx"] or 4 + 5 * i % 9, "nu": case["nu"] or 2 + i % 3}
        out.append((W.mpc_qp(sd, x0_scale=0.5, **size), W.mpc_qp(sd, x0_scale=0.45, **size)))
    return out


def _settings(case):
    st = clr.clr_default_settings(case["bits"])
    if case["kind"] != "qp":
        st.eps_feas = EPS
    if "iters" in case:
        st.max_iter = case["iters"]
    return st


def _dense_system(case, seed):
    """Quasi-definite [H A'; A -G], columns first (column-major), its signs and a right-hand side."""
    n = case["n"]
    rng = np.random.default_rng(seed)
    p = max(1, (2 * n) // 3)
    M = rng.standard_normal((n, n)) / math.sqrt(n)
    K = M + M.T
    H = rng.standard_normal((p, p)) / math.sqrt(p)
    K[:p, :p] = H @ H.T + 0.5 * np.eye(p)
    K[p:, p:] = -np.diag(rng.uniform(0.1, 2.0, n - p))
    return K, np.r_[np.ones(p), -np.ones(n - p)], rng.standard_normal(n)


def _arrays(sol):
    x, s, z, info = sol
    return {"x": x, "s": s, "z": z, "status": info["status"]}


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    k = case["kind"]
    if k == "dense_kkt":
        K, signs, rhs = _dense_system(case, seed)
        dev = torch.device("cuda")
        n = case["n"]
        return {"kind": k, "n": n, "K": torch.tensor(K, device=dev), "signs": torch.tensor(signs, device=dev),
                "rhs": torch.tensor(rhs, device=dev), "x": torch.empty(n, dtype=torch.float64, device=dev),
                "D": torch.empty(n, dtype=torch.float64, device=dev),
                "hits": torch.zeros(1, dtype=torch.int32, device=dev)}
    if k == "mpc":
        pairs = _mpc_pairs(case, seed)
        args = [(a.P, a.q, a.A, a.b, a.cones) for a, _ in pairs]
        new = [(c.q, c.b) for _, c in pairs]
        if case["count"] == 1:
            return {"kind": "update", "solver": clr.clr_setup(*args[0], _settings(case)), "new": new[0]}
        return {"kind": "cohort", "solver": clr.clr_batch_setup(args, _settings(case)), "new": new}
    pr = _problem(case, seed)
    if k == "portfolio":  # set up with last period's expected returns
        rng = np.random.default_rng(seed + 1)
        q0 = pr.q.copy()
        q0[:case["n"]] += 0.1 * rng.standard_normal(case["n"])
        return {"kind": "update", "solver": clr.clr_setup(pr.P, q0, pr.A, pr.b, pr.cones, _settings(case)),
                "new": (pr.q, pr.b)}
    return {"kind": "solve", "solver": clr.clr_setup(pr.P, pr.q, pr.A, pr.b, pr.cones, _settings(case))}


def run(state):
    k = state["kind"]
    if k == "dense_kkt":
        clr.clr_dense_ldl_solve_noalloc(state["K"].data_ptr(), state["signs"].data_ptr(), state["n"],
                                        state["rhs"].data_ptr(), state["x"].data_ptr(), state["D"].data_ptr(),
                                        hits_ptr=state["hits"].data_ptr(),
                                        stream_ptr=torch.cuda.current_stream().cuda_stream)
        return {"x": state["x"], "D": state["D"], "hits": state["hits"]}
    sv = state["solver"]
    if k == "cohort":
        for i, (q, b) in enumerate(state["new"]):
            sv.update_qb_of(i, q, b)
        sv.solve()
        sols = [sv.solution_of(i) for i in range(len(state["new"]))]
        return {"x": np.concatenate([t[0] for t in sols]), "s": np.concatenate([t[1] for t in sols]),
                "z": np.concatenate([t[2] for t in sols]), "status": np.array([t[3]["status"] for t in sols])}
    if k == "update":
        sv.update_qb(*state["new"])
    sv.solve()
    return _arrays(sv.solution())


# ---------------------------------------------------------------- least work
def work(case):
    """Least bytes and flops of one pass: the data in and the answer out once, and per
    factorization the flops of eliminating the problem's own structure (fill of a good
    order), per iteration about three solves with the factor."""
    k = case["kind"]
    if k == "dense_kkt":
        n = case["n"]
        return {"bytes": 8 * (n * (n + 1) // 2 + 4 * n), "flops": n ** 3 / 3 + 4 * n * n}
    if k == "qp":
        n, its = case["n"], 10
        m, nnz, fac, lnz = 2 * n, 2 * n * n, 2 * n * n * n + n ** 3 / 3, 2.5 * n * n
    elif k == "mpc":
        its, c = 6, case["count"]
        T, nx, nu = case["T"] or 30, case["nx"] or 8, case["nu"] or 3
        n, m = c * T * (nx + nu), c * (T * nx + 2 * T * (nx + nu) + T * (nu + 1))
        nnz = c * T * (nx * nx + nx * nu) + m
        fac, lnz = c * T * 4.0 * (2 * nx + nu) ** 3, c * T * 1.5 * (2 * nx + nu) ** 2
    elif k == "mixed":
        n, its = case["n"], case["iters"]
        m = 33 * n // 10
        nnz, fac, lnz = n * n / 2 + 10 * n, n ** 3 / 3, n * n / 2
    elif k == "entropy":
        n0, its = case["n"], case["iters"]
        n, m = 2 * n0, 1 + n0 // 2 + 3 * n0
        nnz, fac, lnz = n0 * n0 // 2 + 3 * n0, n0 * (n0 / 2) ** 2 + (n0 / 2) ** 3 / 3, n0 * n0 / 2 + n0 * n0 / 8
    elif k == "portfolio":
        n, its = case["n"], 12
        p = n // 10
        m, nnz, fac, lnz = n + p + 1, n * p // 2, n * p * p / 4 + p ** 3 / 3, n * p / 2
        n += p
    elif k == "huber":
        n0, its = case["n"], 8
        m0 = 3 * n0 // 2
        n, m = n0 + 3 * m0, 3 * m0
        nnz, fac, lnz = 0.15 * n0 * m0, m0 * (0.15 * n0) ** 2 + n0 ** 3 / 3, 0.15 * n0 * m0 + n0 * n0 / 2
    elif k in ("psd_mixed", "psd_batch"):
        its = case["iters"]
        ks = (2, 3, 4, 5, 8, 10, 16) * case["per_order"] if k == "psd_mixed" else (case["order"],) * (case["n"] // 10)
        n = 30 * case["per_order"] if k == "psd_mixed" else case["n"]
        d = [o * (o + 1) // 2 for o in ks]
        m = sum(d) + n // 4
        nnz = 6 * n
        fac = sum(v ** 3 / 3 + 60.0 * o ** 3 for v, o in zip(d, ks)) + n ** 3 / 3
        lnz = sum(v * v / 2 for v in d) + n * n / 2
    else:
        n, its = case["n"], case["iters"]
        m, nnz, fac, lnz = 2 * n, 8 * n, 6e5 * n, 790 * n
    word = case["bits"] // 8
    return {"bytes": 8.0 * (n + m + nnz) + 8.0 * (n + 2 * m) + its * lnz * word,
            "flops": float(its * (fac + 3 * 4 * lnz))}


# ---------------------------------------------------------------- exact answers
def _ldl(K):
    n = len(K)
    A, D = K.copy(), np.empty(n)
    for j in range(n):
        D[j] = A[j, j]
        col = A[j + 1:, j] / D[j]
        A[j + 1:, j + 1:] -= np.outer(col, A[j, j + 1:])
        A[j + 1:, j] = col
    return D


def _exact_huber(pr):
    """Reweighted least squares, then Newton on the Huber loss (piecewise quadratic: it ends at the
    minimiser of the right piece), then every variable of the conic form."""
    A, b, T = pr.meta["A"].toarray(), pr.meta["b"], pr.meta["T"]
    x = np.zeros(A.shape[1])
    for _ in range(25):
        w = np.minimum(1.0, T / np.maximum(np.abs(A @ x - b), 1e-300))
        x = np.linalg.solve(A.T @ (w[:, None] * A), A.T @ (w * b))
    for _ in range(50):
        r = A @ x - b
        B = A[np.abs(r) <= T]
        step = np.linalg.solve(B.T @ B, A.T @ np.clip(r, -T, T))
        x = x - step
        if np.linalg.norm(step) <= 1e-13 * np.linalg.norm(x):
            break
    else:
        return None
    r = A @ x - b
    u = np.clip(r, -T, T)
    pos, neg = np.maximum(r - T, 0.0), np.maximum(-r - T, 0.0)
    return {"x": np.r_[x, u, pos, neg], "s": np.r_[np.zeros(len(b)), pos, neg],
            "z": np.r_[2 * u, 2 * T - 2 * u, 2 * T + 2 * u], "status": 1}


def _exact_portfolio(pr):
    """Active-set steps on x >= 0 with the low-rank structure, then the conic form's variables."""
    F, d, mu = pr.meta["F"].toarray(), pr.meta["d"], pr.meta["mu"]
    n, p = F.shape
    on = np.ones(n, bool)
    for _ in range(200):
        Fs, di = F[on], 0.5 / d[on]
        C = 0.5 * np.eye(p) + Fs.T @ (di[:, None] * Fs)  # Woodbury on 2 D + 2 F F'

        def inv(v):
            t = di[:, None] * v
            return t - di[:, None] * (Fs @ np.linalg.solve(C, Fs.T @ t))

        h = inv(np.c_[mu[on], np.ones(on.sum())])
        nu = (h[:, 0].sum() - 1.0) / h[:, 1].sum()
        x = np.zeros(n)
        x[on] = h[:, 0] - nu * h[:, 1]
        y = F.T @ x
        z = np.where(on, 0.0, 2 * d * x + 2 * (F @ y) - mu + nu)
        new = x - z > 0
        if np.array_equal(new, on):
            return {"x": np.r_[x, y], "s": np.r_[np.zeros(p + 1), x], "z": np.r_[2 * y, nu, z], "status": 1}
        on = new
    return None


def exact(case, seed):
    k = case["kind"]
    if k == "dense_kkt":
        K, _, rhs = _dense_system(case, seed)
        return {"x": np.linalg.solve(K, rhs), "D": _ldl(K), "hits": np.zeros(1, np.int32)}
    if k == "qp":
        pr = _problem(case, seed)
        return {"x": pr.x_star, "s": pr.s_star, "z": pr.z_star, "status": 1}
    if k == "huber":
        return _exact_huber(_problem(case, seed))
    if k == "portfolio":
        return _exact_portfolio(_problem(case, seed))
    return None
