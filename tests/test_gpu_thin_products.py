"""Many thin leaf fronts under one parent: as a product or by lists, with the path asserted
(clr_ldl_routes)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
clr = pytest.importorskip("paper_2412_19027_gb300.clr")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_19027_gb300 import build
    build.build()


KID = 12


def arrow(leaves, c, r, m, deep=0, few=0, shared=0, seed=0):
    """Cliques of c pivots on r of the m root rows, the first `shared` of them common; `deep` more have a
    child of KID pivots (too many to be merged into them), `few` more only 20 rows.  Quasi-definite,
    diagonally dominant."""
    import scipy.sparse as sp
    rng = np.random.default_rng(seed + leaves + c + r + m)
    R, Cc, V, p0 = [], [], [], 0
    kinds = rng.permutation(np.r_[np.zeros(leaves, int), np.ones(deep, int), np.full(few, 2)])
    root = leaves * c + deep * (c + KID) + few * c
    N = root + m
    for kind in kinds:
        piv = np.arange(p0, p0 + c + (KID if kind == 1 else 0))
        p0 += len(piv)
        for a in piv:
            low = piv[piv > a]
            R.append(low); Cc.append(np.full(len(low), a)); V.append(0.1 * rng.standard_normal(len(low)))
        rr = 20 if kind == 2 else r
        sh = min(shared, rr)
        rows = root + np.r_[np.arange(sh), sh + np.sort(rng.choice(m - sh, rr - sh, replace=False))]
        for a in piv[-c:]:
            R.append(rows); Cc.append(np.full(rr, a)); V.append(rng.standard_normal(rr) / np.sqrt(len(kinds) * r))
    K = sp.csc_matrix((np.concatenate(V), (np.concatenate(R), np.concatenate(Cc))), shape=(N, N))
    sgn = np.where(np.arange(N) < root, 1.0, -1.0)
    return sp.csc_matrix(sp.tril(K, -1) + sp.diags(sgn * (2.0 + rng.random(N)))), sgn, rng.standard_normal(N)


def check(K, sgn, rhs, bits):
    import scipy.sparse as sp
    N = len(rhs)
    x, D, hits = clr.clr_ldl_solve(K, sgn, rhs, order=np.arange(N), factor_bits=bits)
    Kf = K + sp.tril(K, -1).T
    # diagonally dominant quasi-definite blocks, growth < 10: backward error of the order of (sources + rows) eps
    eps = 2.2e-16 if bits == 64 else 1.2e-7
    assert np.abs(Kf @ x - rhs).max() <= 10 * np.sqrt(N) * eps * max(1.0, np.abs(x).max()) * 10
    assert hits == 0 and np.all(sgn * D > 0)


# 512 leaves besides the four that the parent takes by relative indices and those that are merged into
# it; several pivots a leaf (their diagonal block's solves, more columns than leaves)
@pytest.mark.parametrize("bits,leaves,c,r,m,deep,few", [
    (32, 530, 2, 130, 200, 0, 0), (32, 560, 3, 190, 193, 5, 0), (32, 560, 16, 140, 150, 0, 4), (32, 570, 5, 129, 300, 2, 3),
    (32, 620, 1, 256, 400, 0, 0), (64, 570, 1, 150, 185, 0, 0), (64, 650, 1, 190, 240, 3, 3), (64, 1100, 1, 257, 320, 0, 0)])
def test_product_of_thin_leaves(bits, leaves, c, r, m, deep, few):
    K, sgn, rhs = arrow(leaves, c, r, m, deep, few)
    got = clr.clr_ldl_routes(K, order=np.arange(len(rhs)), factor_bits=bits)
    assert got["product_parents"] == 1 and got["product_leaves"] >= 512
    check(K, sgn, rhs, bits)


# thin fronts by lists: too many zeros in the product's panel, or too few leaves of the parent beside fronts
# with children; lists of more than 512 sources (a warp) and of more than 8192 (a CTA)
@pytest.mark.parametrize("bits,leaves,c,r,m,deep,few,shared,warps,ctas", [
    (64, 2500, 1, 110, 165, 0, 0, 0, 1, 0), (64, 9000, 1, 100, 152, 0, 0, 20, 1, 1), (64, 600, 16, 140, 150, 20, 0, 0, 1, 0),
    (64, 530, 5, 150, 200, 520, 0, 0, 1, 0), (32, 300, 5, 129, 250, 300, 2, 0, 0, 0), (32, 10, 16, 129, 200, 560, 0, 0, 0, 0),
    (64, 10, 1, 129, 220, 560, 0, 0, 0, 0)])
def test_thin_fronts_by_lists(bits, leaves, c, r, m, deep, few, shared, warps, ctas):
    K, sgn, rhs = arrow(leaves, c, r, m, deep, few, shared)
    got = clr.clr_ldl_routes(K, order=np.arange(len(rhs)), factor_bits=bits)
    assert got["product_parents"] == 0 and got["thin_fronts"] >= 512
    assert (got["warp_lists"] > 0) == bool(warps) and (got["cta_lists"] > 0) == bool(ctas)
    check(K, sgn, rhs, bits)


# a leaf whose pivot overflows in FP32: its column of L is zero and takes nothing off its parent, by lists (too
# many zeros for the product) and by the product
@pytest.mark.parametrize("r,m,parents", [(129, 1100, 0), (140, 200, 1)])
def test_infinite_pivot_of_a_leaf(r, m, parents):
    import scipy.sparse as sp
    K, sgn, rhs = arrow(560, 1, r, m)
    N = len(rhs)
    got = clr.clr_ldl_routes(K, order=np.arange(N), factor_bits=32)
    assert got["product_parents"] == parents and got["thin_fronts"] >= 512
    K = K.tolil()
    K[7, 7] = 1e39
    x, D, hits = clr.clr_ldl_solve(sp.csc_matrix(K), sgn, rhs, order=np.arange(N), factor_bits=32)
    assert np.isinf(D[7]) and x[7] == 0 and np.all(np.isfinite(x)) and np.all(np.isfinite(np.delete(D, 7)))
    Kf = sp.csc_matrix(K + sp.tril(K, -1).T)
    r = (Kf @ x - rhs)[np.arange(N) != 7]
    assert np.abs(r).max() <= 10 * np.sqrt(N) * 1.2e-7 * max(1.0, np.abs(x).max()) * 10


# with an escalation to FP64 possible, a plan that FP64 would pay for stays with the lists (23 FMAs of the
# product per value); without it, and at half the zeros (8.5), the product is taken
@pytest.mark.parametrize("density,escalation,parents", [(0.3, 1, 0), (0.3, 0, 1), (0.5, 1, 1)])
def test_product_of_a_solver_that_may_escalate(density, escalation, parents):
    from paper_2412_19027_gb300 import workloads as W
    p = W.portfolio_qp(1, n=5000, density=density)
    st = clr.clr_default_settings(32, max_iter=2, fp64_escalation=escalation)
    sv = clr.clr_setup(p.P, p.q, p.A, p.b, p.cones, st)
    assert sv.routes()["product_parents"] == parents
    sv.free()
