"""Dense QPs with a unique, nondegenerate optimum on both sides of the sizes at which the factorization's
kernels change (FP64 fronts of more than 320 rows: products by digits; 512 thin fronts: k_factor_thin; lists
of more than 512 sources: summed by trees): one error bound for all, from the termination tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
clr = pytest.importorskip("paper_2412_19027_gb300.clr")
from paper_2412_19027_gb300 import workloads as W  # noqa: E402

EPS = 1e-8


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2412_19027_gb300 import build
    build.build()


# At termination the residuals are below EPS times their norms and the gap, sum of s z, below EPS max(1,
# |objective|).  At the optimum s and z are >= 1/2 where they are not zero (unique_qp), so the inactive rows
# keep sum z <= 2 gap and the active ones |s| <= 2 gap.  All of it is a perturbation of the right-hand side of
# [P A'; A 0] over the active rows, and the solution moves by its 2-norm over the smallest singular value.
@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("n", [200, 240, 255, 270, 300, 520])
def test_optimum_on_both_sides_of_the_kernel_limits(bits, n):
    import scipy.sparse as sp
    p = W.unique_qp(n, n=n, n_eq=n // 5, n_inactive=n, rank=5)
    sv = clr.clr_setup(p.P, p.q, p.A, p.b, p.cones, clr.clr_default_settings(bits))
    sv.solve()
    x, s, z, info = sv.solution()
    routes, sym = sv.routes(), sv.symbolic()
    sv.free()
    f, c = np.diff(sym["row_ptr"]), np.diff(sym["sn_ptr"])
    assert routes["digit_fronts"] == (np.sum((f > 320) & (c > 8)) if bits == 64 else 0)
    assert info["status_name"] == "SOLVED"
    P = p.P.toarray()
    P = np.triu(P) + np.triu(P, 1).T
    A = sp.csr_matrix(p.A).toarray()
    act = p.s_star == 0
    K = np.block([[P, A[act].T], [A[act], np.zeros((act.sum(), act.sum()))]])
    smin = np.linalg.svd(K, compute_uv=False)[-1]
    inf = lambda v: np.abs(v).max()
    rd = max(1.0, inf(P @ p.x_star), inf(A.T @ p.z_star), inf(p.q))
    rp = max(1.0, inf(p.b) + inf(p.x_star) + inf(p.s_star))
    gap = EPS * max(1.0, abs(0.5 * p.x_star @ P @ p.x_star + p.q @ p.x_star))
    row = np.linalg.norm(A, axis=1).max()
    bound = (np.sqrt(len(K)) * EPS * (rd + rp) + 2 * gap * (1 + row)) / smin
    assert np.linalg.norm(np.r_[x - p.x_star, (z - p.z_star)[act]]) <= bound
