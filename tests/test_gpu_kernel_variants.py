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
