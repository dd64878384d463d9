"""Kernel variants chosen by size: each against the general path or the oracle, at
the sizes where its tiles, lanes or lists end."""
import numpy as np
import pytest

from oracle import cones as OC
from oracle.linsys import ldl_factor, ldl_solve

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
clr = pytest.importorskip("paper_2412_19027_gb300.clr")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_19027_gb300 import build
    build.build()


# the register tiles of the dense solve hold N + 1 rows in steps of 16; 48 KB of
# shared memory hold L up to N = 110
@pytest.mark.parametrize("N", [1, 2, 15, 16, 17, 31, 33, 47, 48, 63, 64, 95, 96, 107, 111, 112, 127, 128])
def test_dense_ldl_tile_edges(N):
    rng = np.random.default_rng(N)
    p = max(1, (2 * N) // 3)
    K = rng.standard_normal((N, N)) / np.sqrt(N)
    K = K + K.T
    H = rng.standard_normal((p, p)) / np.sqrt(p)
    K[:p, :p] = H @ H.T + 0.5 * np.eye(p)
    K[p:, p:] = -np.diag(rng.uniform(0.1, 2.0, N - p))
    signs, rhs = np.r_[np.ones(p), -np.ones(N - p)], rng.standard_normal(N)
    dev = torch.device("cuda")
    Kd = torch.tensor(np.tril(K) + np.triu(np.full_like(K, np.nan), 1), device=dev).t().contiguous()
    sd, bd = torch.tensor(signs, device=dev), torch.tensor(rhs, device=dev)
    x, D = torch.empty(N, dtype=torch.float64, device=dev), torch.empty(N, dtype=torch.float64, device=dev)
    hits = torch.full((1,), -1, dtype=torch.int32, device=dev)
    clr.clr_dense_ldl_solve_noalloc(Kd.data_ptr(), sd.data_ptr(), N, bd.data_ptr(), x.data_ptr(), D.data_ptr(),
                                    hits_ptr=hits.data_ptr(), stream_ptr=torch.cuda.current_stream().cuda_stream)
    L, Dref, _ = ldl_factor(K, signs, 1e-13, 2e-7)
    x, D = x.cpu().numpy(), D.cpu().numpy()
    # unpivoted LDL of a quasi-definite matrix with unit-sized blocks: errors of N eps times its growth (< 1e3)
    np.testing.assert_allclose(D, Dref, rtol=N * 2.2e-16 * 1e3)
    xref = ldl_solve(L, Dref, rhs)
    assert np.abs(K @ x - rhs).max() <= N * 2.2e-16 * 1e3 * max(1.0, np.abs(xref).max())
    assert int(hits.item()) == 0


# PSD step length: lanes per cone for short lists, a thread per cone for long ones; same bits
@pytest.mark.parametrize("orders", [(1, 2, 3, 4), (5, 6, 7, 8), (9, 12, 15, 16)])
def test_psd_step_lane_equals_thread(orders):
    rng = np.random.default_rng(sum(orders))
    cones, s, z, ds, dz = [], [], [], [], []
    for rep in range(5):
        for k in orders:
            cones.append((OC.PSD, k * (k + 1) // 2, 0.0))
            for out in (s, z):
                M = rng.standard_normal((k, k))
                out.append(OC.svec(M @ M.T / k + 0.3 * np.eye(k)))
            for out in (ds, dz):
                T = rng.standard_normal((k, k))
                out.append(OC.svec(T + T.T) if rep else OC.svec(np.diag(rng.uniform(0.1, 1.0, k))))
    ref = []
    for i in range(len(cones)):  # every cone on its own, against the oracle
        a = clr.clr_cones_step_length([cones[i]], s[i], z[i], ds[i], dz[i], 1e6)
        o = min(1e6, OC.step_length_symmetric(OC.PSD, s[i], ds[i]), OC.step_length_symmetric(OC.PSD, z[i], dz[i]))
        assert a == pytest.approx(o, rel=1e-10)
        ref.append(a)
    reps = 4096 // len(cones) + 1  # longer than the list length up to which lanes are used
    for i in (0, len(cones) - 1, int(np.argmin(ref))):
        many = clr.clr_cones_step_length([cones[i]] * (4097), np.tile(s[i], 4097), np.tile(z[i], 4097),
                                         np.tile(ds[i], 4097), np.tile(dz[i], 4097), 1e6)
        assert many == ref[i]
    cat = lambda v, r: np.tile(np.concatenate(v), r)
    few = clr.clr_cones_step_length(cones, *[cat(v, 1) for v in (s, z, ds, dz)], 1e6)
    many = clr.clr_cones_step_length(cones * reps, *[cat(v, reps) for v in (s, z, ds, dz)], 1e6)
    assert few == many == min(ref)


# fronts of few pivots and many rows (k_factor_thin) and long pull lists: an arrow matrix
# of `leaves` cliques of c pivots on r of the m root rows (leaf fronts of c + r rows)
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("leaves,c,r,m,extra", [
    (3, 1, 130, 140, 0), (60, 2, 129, 200, 0), (60, 3, 192, 260, 4), (700, 1, 191, 193, 0),
    (49, 16, 300, 330, 0), (20, 5, 256, 300, 9), (9000, 1, 128, 129, 0), (6, 17, 140, 160, 0)])
def test_thin_fronts_and_long_pulls(bits, leaves, c, r, m, extra):
    import scipy.sparse as sp
    rng = np.random.default_rng(leaves + r)
    N = leaves * (c + extra) + m
    R, Cc, V = [], [], []
    root = N - m
    # with extra: a first clique of `extra` pivots under each leaf, so that the thin front has a child
    for q in range(leaves):
        p0 = q * (c + extra)
        piv = np.arange(p0, p0 + extra + c)
        for a in piv:
            low = piv[piv > a]
            R += list(low); Cc += [a] * len(low); V += list(0.1 * rng.standard_normal(len(low)))
        rows = root + np.sort(rng.choice(m, r, replace=False))
        for a in piv[extra:]:
            R += list(rows); Cc += [a] * r; V += list(rng.standard_normal(r) / np.sqrt(leaves * r))
    K = sp.csc_matrix((V, (R, Cc)), shape=(N, N))
    sgn = np.where(np.arange(N) < root, 1.0, -1.0)
    K = sp.tril(K, -1) + sp.diags(sgn * (2.0 + rng.random(N)))
    rhs = rng.standard_normal(N)
    x, D, hits = clr.clr_ldl_solve(K, sgn, rhs, order=np.arange(N), factor_bits=bits)
    Kf = K + sp.tril(K, -1).T
    # diagonally dominant quasi-definite blocks, growth < 10: backward error of the order of (sources + rows) eps
    eps = 2.2e-16 if bits == 64 else 1.2e-7
    assert np.abs(Kf @ x - rhs).max() <= 10 * np.sqrt(N) * eps * max(1.0, np.abs(x).max()) * 10
    assert hits == 0 and np.all(sgn * D > 0)


# 512 thin leaves or more under one parent: their update matrices as one product (thinsyrk.cu), at
# the ends of its 64 x 64 tiles, 16-column steps and splits; `deep` leaves have a child and `few`
# have too few rows to be thin, and stay with the lists beside it
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("leaves,c,r,m,deep,few", [
    (512, 1, 129, 129, 0, 0), (515, 1, 128, 192, 0, 0), (530, 1, 190, 193, 9, 0), (513, 2, 130, 255, 0, 5),
    (600, 1, 256, 256, 3, 3), (512, 3, 257, 257, 0, 0), (2100, 1, 140, 140, 0, 7), (511, 1, 130, 130, 2, 2)])
def test_thin_leaves_as_product(bits, leaves, c, r, m, deep, few):
    import scipy.sparse as sp
    rng = np.random.default_rng(leaves + c + r + m)
    R, Cc, V, p0 = [], [], [], 0
    kinds = rng.permutation(np.r_[np.zeros(leaves, int), np.ones(deep, int), np.full(few, 2)])
    root = leaves * c + deep * (c + 3) + few * c
    N = root + m
    for kind in kinds:
        piv = np.arange(p0, p0 + c + (3 if kind == 1 else 0))
        p0 += len(piv)
        for a in piv:
            low = piv[piv > a]
            R.append(low); Cc.append(np.full(len(low), a)); V.append(0.1 * rng.standard_normal(len(low)))
        rr = 20 if kind == 2 else r
        rows = root + np.sort(rng.choice(m, rr, replace=False))
        for a in piv[-c:]:
            R.append(rows); Cc.append(np.full(rr, a)); V.append(rng.standard_normal(rr) / np.sqrt(len(kinds) * r))
    K = sp.csc_matrix((np.concatenate(V), (np.concatenate(R), np.concatenate(Cc))), shape=(N, N))
    sgn = np.where(np.arange(N) < root, 1.0, -1.0)
    K = sp.tril(K, -1) + sp.diags(sgn * (2.0 + rng.random(N)))
    rhs = rng.standard_normal(N)
    x, D, hits = clr.clr_ldl_solve(K, sgn, rhs, order=np.arange(N), factor_bits=bits)
    Kf = K + sp.tril(K, -1).T
    # as above: diagonally dominant quasi-definite blocks
    eps = 2.2e-16 if bits == 64 else 1.2e-7
    assert np.abs(Kf @ x - rhs).max() <= 10 * np.sqrt(N) * eps * max(1.0, np.abs(x).max()) * 10
    assert hits == 0 and np.all(sgn * D > 0)


# one CTA per problem (fronts of at most 96 rows, all of a cohort) against the launch per
# level: the same problem alone and beside one with large fronts, which takes every problem
# of the cohort through the general kernels
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("make", [
    lambda W: W.mpc_qp(1, T=10, nx=4, nu=2), lambda W: W.mpc_qp(2, T=50, nx=12, nu=4),
    lambda W: W.mpc_qp(3, T=31, nx=5, nu=3), lambda W: W.unique_qp(4, n=10, n_eq=2, n_inactive=10),
    lambda W: W.unique_qp(5, n=30, n_eq=6, n_inactive=30), lambda W: W.unique_qp(6, n=50, n_eq=10, n_inactive=50),
    lambda W: W.unique_qp(7, n=68, n_eq=4, n_inactive=30), lambda W: W.psd_mixed(8, orders=(2, 3, 4), per_order=2)])
def test_cta_solves_equal_level_launches(bits, make):
    from paper_2412_19027_gb300 import workloads as W
    pr, big = make(W), W.mixed_cone(9, n=300, n_zero=0, n_nonneg=525, n_soc=75, n_exp=15, n_pow=15)
    st = clr.clr_default_settings(bits, max_iter=6, fp64_escalation=0)
    arg = lambda p: (p.P, p.q, p.A, p.b, p.cones)
    one = clr.clr_setup(*arg(pr), st)
    one.solve()
    both = clr.clr_batch_setup([arg(pr), arg(big)], st)
    both.solve()
    a, b = one.solution(), both.solution_of(0)
    for u, v in zip(a[:3], b[:3]):
        np.testing.assert_array_equal(u, v)
    assert a[3]["iterations"] == b[3]["iterations"] and a[3]["ir_steps_total"] == b[3]["ir_steps_total"]
    one.free()
    both.free()


# the sweeps over large fronts (k_sweep_fwd up to 512 pivots, k_sweep_bwd) at the ends of
# their batches and prefetches, one front by value and more than four from the list: leaf
# cliques of c pivots on r of the m root rows
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("leaves,c,r,m", [
    (1, 512, 33, 160), (1, 513, 40, 160), (2, 511, 1025, 1030), (5, 129, 1023, 1100), (6, 128, 31, 140),
    (4, 257, 64, 200), (9, 97, 130, 140), (1, 121, 1056, 1060)])
def test_large_front_sweeps(bits, leaves, c, r, m):
    import scipy.sparse as sp
    rng = np.random.default_rng(leaves + c + r)
    N, R, Cc, V = leaves * c + m, [], [], []
    root = N - m
    for q in range(leaves):
        p0 = q * c
        low = np.tril_indices(c, -1)
        R.append(p0 + low[0]); Cc.append(p0 + low[1]); V.append(rng.standard_normal(len(low[0])) / c)
        rows = root + np.sort(rng.choice(m, r, replace=False))
        R.append(np.tile(rows, c)); Cc.append(np.repeat(np.arange(p0, p0 + c), r))
        V.append(rng.standard_normal(c * r) / np.sqrt(c * r))
    low = np.tril_indices(m, -1)
    R.append(root + low[0]); Cc.append(root + low[1]); V.append(rng.standard_normal(len(low[0])) / m)
    K = sp.csc_matrix((np.concatenate(V), (np.concatenate(R), np.concatenate(Cc))), shape=(N, N))
    sgn = np.where(np.arange(N) < root, 1.0, -1.0)
    K = sp.tril(K, -1) + sp.diags(sgn * (2.0 + rng.random(N)))
    rhs = rng.standard_normal(N)
    x, D, hits = clr.clr_ldl_solve(K, sgn, rhs, order=np.arange(N), factor_bits=bits)
    Kf = K + sp.tril(K, -1).T
    # well conditioned (diagonally dominant blocks): rows of up to c + r terms of size <= 1
    eps = 2.2e-16 if bits == 64 else 1.2e-7
    assert np.abs(Kf @ x - rhs).max() <= 10 * np.sqrt(N) * eps * max(1.0, np.abs(x).max()) * 10
    assert hits == 0 and np.all(sgn * D > 0)


# FP64 fronts of more than 320 rows with products of 8-bit digits on the tensor cores, at the ends
# of their 64-row blocks, against FMA products (schedule 2).  Per entry the residual of a solve
# by computed factors is below 3 n u |L||D||L^T||x| (Higham, "Accuracy and Stability of Numerical
# Algorithms", ch. 10), with rows and columns scaled by powers of ten as well; the inverses of the
# diagonal blocks add their condition (here below 10).
@pytest.mark.parametrize("scale", [0, 60])
@pytest.mark.parametrize("n", [320, 321, 383, 384, 385, 449, 512, 639])
def test_large_fp64_fronts_by_digits(n, scale):
    import scipy.sparse as sp
    rng = np.random.default_rng(n + scale)
    p = 2 * n // 3
    K = rng.standard_normal((n, n)) / np.sqrt(n)
    K = K + K.T
    H, G = rng.standard_normal((p, p)) / np.sqrt(p), rng.standard_normal((n - p, n - p)) / np.sqrt(n - p)
    K[:p, :p], K[p:, p:] = H @ H.T + 0.1 * np.eye(p), -(G @ G.T + 0.1 * np.eye(n - p))
    q = rng.permutation(n)  # both signs in every block
    K, sgn = K[np.ix_(q, q)], np.where(q < p, 1.0, -1.0)
    s = 10.0 ** np.round(rng.uniform(-scale, scale, n))
    K, rhs = K * s[:, None] * s[None, :], rng.standard_normal(n) * s
    L, D = np.tril(K).astype(np.float64), np.zeros(n)
    for j in range(n):
        D[j] = L[j, j]
        c = L[j + 1:, j] / D[j]
        L[j + 1:, j + 1:] -= np.tril(np.outer(c, L[j + 1:, j]))
        L[j + 1:, j], L[j, j] = c, 1.0
    res = {}
    for sch in (1, 2):
        x, Dg, hits = clr.clr_ldl_solve(sp.csc_matrix(np.tril(K)), sgn, rhs, order=np.arange(n), dyn_reg_eps=0.0,
                                        big_front_schedule=sch)
        bound = 3 * n * 2.0 ** -53 * (np.abs(L) @ (np.abs(D)[:, None] * (np.abs(L).T @ np.abs(x)[:, None])))[:, 0]
        r = np.abs((rhs.astype(np.longdouble) - K.astype(np.longdouble) @ x).astype(np.float64))
        assert np.all(r <= 10 * bound)
        assert hits == 0 and np.all(sgn * Dg > 0)
        np.testing.assert_allclose(Dg, D, rtol=1e-10)
        res[sch] = np.linalg.norm(r / s)
    assert res[1] <= 2 * res[2]


# K products by row length in one launch (k_kmv_rows: thread, warp and CTA per row) against the lane
# groups: a problem of dense rows alone, and beside a sparse one that brings the rows' average
# down; P and A columns of every length around the limits, a SOC block beside the nonnegative rows
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("n", [130, 520, 700])
def test_k_products_by_row_length(bits, n):
    import scipy.sparse as sp
    from paper_2412_19027_gb300 import workloads as W
    rng = np.random.default_rng(n)
    lens = [1, 2, 3, 4, 5, 31, 32, 33, 127, 128, 129] + [k for k in (509, 510, 511, 512, 513, 514, 641) if k <= n] + [n] * 40
    R = np.concatenate([np.full(k, i) for i, k in enumerate(lens)])
    Cc = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens])
    A = sp.csc_matrix((rng.standard_normal(len(R)) / np.sqrt(n), (R, Cc)), shape=(len(lens), n))
    m = len(lens)
    P, q = sp.csc_matrix(sp.diags(1.0 + rng.random(n))), rng.standard_normal(n)
    s0 = np.r_[1.0 + rng.random(m - 12), 5.0, 0.1 * rng.standard_normal(11)]
    dense = (P, q, A, A @ rng.standard_normal(n) + s0, [(W.NONNEG, m - 12, 0.0), (W.SOC, 12, 0.0)])
    big = W.banded_lp(3, n=6000)
    st = clr.clr_default_settings(bits, max_iter=5, fp64_escalation=0)
    one = clr.clr_setup(*dense, st)
    one.solve()
    both = clr.clr_batch_setup([dense, (big.P, big.q, big.A, big.b, big.cones)], st)
    both.solve()
    a, b = one.solution(), both.solution_of(0)
    for u, v in zip(a[:3], b[:3]):
        np.testing.assert_array_equal(u, v)
    assert a[3]["iterations"] == b[3]["iterations"] and a[3]["ir_steps_total"] == b[3]["ir_steps_total"]
    one.free()
    both.free()


# the panels of thin leaves in solvers built while others run (stream-ordered memory, reused from one
# solver to the next): the server's results are those of a solver built alone
@pytest.mark.parametrize("bits", [64, 32])
def test_thin_leaf_panels_in_server(bits):
    from paper_2412_19027_gb300 import workloads as W
    st = clr.clr_default_settings(bits, max_iter=40)
    arg = lambda p: (p.P, p.q, p.A, p.b, p.cones)
    probs = [W.portfolio_qp(k, n=1500 + 700 * k, density=1.0) for k in (0, 1, 0, 1)]
    sv = clr.Server(device_bytes=8 << 30, max_cohort=1, max_active=2, settings=st)
    reqs = [clr.Request(*arg(p)) for p in probs]
    tickets = [sv.submit(r) for r in reqs]
    got = [sv.wait(t, 120.0) for t in tickets]
    sv.close()
    for p, g in zip(probs, got):
        s = clr.clr_setup(*arg(p), st)
        s.solve()
        want = s.solution()
        for u, v in zip(want[:3], g[:3]):
            np.testing.assert_array_equal(u, v)
        assert want[3]["iterations"] == g[3]["iterations"]
        s.free()
