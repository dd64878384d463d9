"""Which kernels a problem takes (Solver.routes) where the choice is one of time, and that both
sides of a choice give the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
clr = pytest.importorskip("paper_2412_19027_gb300.clr")
from paper_2412_19027_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_19027_gb300 import build
    build.build()


def arg(p):
    return p.P, p.q, p.A, p.b, p.cones


def separable(n, seed=0):
    """min x'Px/2 + q'x, |x| <= 1: n independent fronts of three rows."""
    import scipy.sparse as sp
    rng = np.random.default_rng(seed)
    return (sp.csc_matrix(sp.diags(rng.random(n) + 0.1)), rng.standard_normal(n),
            sp.csc_matrix(sp.vstack([sp.eye(n), -sp.eye(n)])), np.ones(2 * n), [(W.NONNEG, 2 * n, 0.0)])


def qp(seed, n):
    return arg(W.unique_qp(seed, n=n, n_eq=n // 5, n_inactive=n, rank=5))


# refined solves by one CTA per problem: chains of small fronts and cohorts of small problems, not one
# problem of thousands of independent fronts or with one large front
@pytest.mark.parametrize("make,one", [
    (lambda: [separable(2000)], 0), (lambda: [separable(40)], 1), (lambda: [qp(1, 70)], 0), (lambda: [qp(1, 20)], 1),
    (lambda: [qp(k, 50) for k in range(64)], 1), (lambda: [arg(W.mpc_qp(1, T=20, nx=8, nu=3))], 1),
    (lambda: [separable(1000, k) for k in range(100)], 1)])
def test_one_cta_solves_where_they_are_faster(make, one):
    sv = clr.clr_batch_setup(make(), clr.clr_default_settings(64, max_iter=2))
    assert sv.routes()["one_cta"] == one
    sv.free()


# a dense QP alone (launches per level) and among 64 (one CTA each): its 65-row front on either path
@pytest.mark.parametrize("bits", [64, 32])
def test_one_cta_in_a_cohort_equals_launches_alone(bits):
    probs = [qp(k, 50) for k in range(64)]
    st = clr.clr_default_settings(bits, max_iter=6, fp64_escalation=0)
    many = clr.clr_batch_setup(probs, st)
    many.solve()
    assert many.routes()["one_cta"] == 1
    for k in (0, 13, 63):
        one = clr.clr_setup(*probs[k], st)
        one.solve()
        assert one.routes()["one_cta"] == 0
        a, b = one.solution(), many.solution_of(k)
        for u, v in zip(a[:3], b[:3]):
            np.testing.assert_array_equal(u, v)
        assert a[3]["ir_steps_total"] == b[3]["ir_steps_total"]
        one.free()
    many.free()


# levels of more than 304 fronts of at most 16 rows (a warp each) against the kernel that takes a CTA
# per front, beside a problem with larger fronts on the same level
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("n", [303, 304, 305, 311, 2000])
def test_tiny_fronts_a_warp_each(bits, n):
    st = clr.clr_default_settings(bits, max_iter=5, fp64_escalation=0)
    big = arg(W.mixed_cone(9, n=300, n_zero=0, n_nonneg=525, n_soc=75, n_exp=15, n_pow=15))
    one = clr.clr_setup(*separable(n), st)
    one.solve()
    both = clr.clr_batch_setup([separable(n), big], st)
    both.solve()
    a, b = one.solution(), both.solution_of(0)
    for u, v in zip(a[:3], b[:3]):
        np.testing.assert_array_equal(u, v)
    one.free()
    both.free()


# forward sweeps of large fronts with the children's gather inside (few CTAs on a level) and apart (a cohort
# whose roots share a level of more than 304)
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("n,count", [(200, 44), (133, 62)])
def test_sweeps_with_and_without_the_gather(bits, n, count):
    import scipy.sparse as sp
    probs = []
    for k in range(count):
        rng = np.random.default_rng(k)
        H = rng.standard_normal((n, n)) / np.sqrt(n)
        A = sp.csc_matrix(sp.vstack([sp.eye(n), -sp.eye(n)]))
        probs.append((sp.csc_matrix(np.triu(H @ H.T + 0.1 * np.eye(n))), rng.standard_normal(n), A, np.ones(2 * n),
                      [(W.NONNEG, 2 * n, 0.0)]))
    st = clr.clr_default_settings(bits, max_iter=4, fp64_escalation=0)
    many = clr.clr_batch_setup(probs, st)
    many.solve()
    for k in (0, count - 1):
        one = clr.clr_setup(*probs[k], st)
        one.solve()
        a, b = one.solution(), many.solution_of(k)
        for u, v in zip(a[:3], b[:3]):
            np.testing.assert_array_equal(u, v)
        one.free()
    many.free()


# FP64 fronts of more than 320 rows: products by digits from 9 pivots on
@pytest.mark.parametrize("c,digits", [(8, 0), (9, 1)])
def test_digit_products_from_9_pivots(c, digits):
    import scipy.sparse as sp
    rng = np.random.default_rng(c)
    m, r, groups = 500, 330, 12  # groups of c coupled variables, each on r rows of one dense second-order cone
    R, Cc, V = [], [], []
    for g in range(groups):
        rows = np.sort(rng.choice(m, r, replace=False))
        for k in range(c):
            R.append(rows); Cc.append(np.full(r, g * c + k)); V.append(rng.standard_normal(r) / np.sqrt(r))
    A = sp.csc_matrix((np.concatenate(V), (np.concatenate(R), np.concatenate(Cc))), shape=(m, groups * c))
    P = sp.csc_matrix(sp.triu(sp.block_diag([sp.coo_matrix(np.eye(c) + 0.05 * np.ones((c, c)))] * groups)))
    st = clr.clr_default_settings(64, max_iter=3, soc_expand_dim=0)
    sv = clr.clr_setup(P, rng.standard_normal(groups * c), A, np.r_[60.0, 0.5 * rng.standard_normal(m - 1)],
                       [(W.SOC, m, 0.0)], st)
    sv.solve()
    sym = sv.symbolic()
    f, p = np.diff(sym["row_ptr"]), np.diff(sym["sn_ptr"])
    got = sv.routes()
    assert got["digit_fronts"] == np.sum((f > 320) & (p > 8)) and (np.sum((f > 320) & (p == c)) > 0)
    assert got["digit_fronts"] < got["big_fronts"] or digits
    assert np.all(np.isfinite(sv.solution()[0]))
    sv.free()


# the autotuner times FMA products (schedule 2) beside digits where an FP64 problem has fronts in digits: three
# amalgamations, four front sizes, three schedules
def test_autotuner_times_fma_products():
    import scipy.sparse as sp
    n = 340
    rng = np.random.default_rng(1)
    H = rng.standard_normal((n, n)) / np.sqrt(n)
    A = sp.csc_matrix(sp.vstack([sp.eye(n), -sp.eye(n)]))
    prob = (sp.csc_matrix(np.triu(H @ H.T + 0.1 * np.eye(n))), rng.standard_normal(n), A, np.ones(2 * n),
            [(W.NONNEG, 2 * n, 0.0)])
    r = clr.clr_autotune([prob], clr.clr_default_settings(64), iters=1)
    assert r["candidates"] == 36
    assert clr.clr_autotune([qp(1, 20)], clr.clr_default_settings(64), iters=1)["candidates"] == 24
