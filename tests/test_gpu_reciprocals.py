"""The reciprocals of the pivot chains against 1.0 / d, through entry points whose second pivot is
-1 / d of the first: [[d, 1], [1, 0]] = L diag(d, -1/d) L'."""
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


def values(k):
    """Mantissas at and beside 1 and 2, all over between; every binade near the limits of the fast path."""
    rng = np.random.default_rng(0)
    one = 1.0 + np.spacing(1.0) * np.r_[np.arange(8), 2.0 ** np.arange(3, 30)]
    two = 2.0 - np.spacing(1.0) * np.r_[np.arange(1, 8), 2.0 ** np.arange(3, 30)]
    mant = np.r_[one, two, rng.uniform(1.0, 2.0, 400)]
    edge = np.array([-1021, -1020, -965, -964, -963, -962, 961, 962, 963, 964, 1019, 1020, 1021])
    ex = np.r_[0, -1, 1, rng.integers(-950, 950, k), edge]
    d = np.concatenate([np.ldexp(mant, int(e)) for e in ex])
    d = d[(1.0 / d > 2.3e-308)]  # (a subnormal pivot is not kept to the last bit)
    return d * np.where(rng.random(len(d)) < 0.5, -1.0, 1.0)


# one unit in the last place of the correctly rounded reciprocal (a final rounding on top of a value that is
# good to 2^-57)
def test_reciprocal_of_the_dense_entry_point():
    d = values(3)[::7]
    dev = torch.device("cuda")
    sg = np.sign(d)
    K = np.zeros((len(d), 2, 2))
    K[:, 0, 0], K[:, 0, 1], K[:, 1, 0] = d, 1.0, 1.0
    Kd, sd = torch.tensor(K, device=dev), torch.tensor(np.stack([sg, -sg], 1), device=dev)
    rhs, x = torch.ones(2, dtype=torch.float64, device=dev), torch.empty(2, dtype=torch.float64, device=dev)
    D = torch.empty((len(d), 2), dtype=torch.float64, device=dev)
    st = torch.cuda.current_stream().cuda_stream
    for i in range(len(d)):
        clr.clr_dense_ldl_solve_noalloc(Kd[i].data_ptr(), sd[i].data_ptr(), 2, rhs.data_ptr(), x.data_ptr(),
                                        D[i].data_ptr(), dyn_reg_eps=0.0, stream_ptr=st)
    got = D.cpu().numpy()
    assert np.array_equal(got[:, 0], d)
    ref = -1.0 / d
    assert np.all(np.abs(got[:, 1] - ref) <= np.spacing(np.abs(ref)))


# the same in one dense FP64 front (explicit zeros outside the blocks), schedule 1: digit products
def test_reciprocal_of_large_fp64_fronts():
    import scipy.sparse as sp
    n = 512
    low = np.nonzero(np.tril(np.ones((n, n), bool)))
    d = values(3)
    rng = np.random.default_rng(1)
    for block in np.array_split(rng.permutation(d), -(-len(d) // (n // 2))):
        block = np.resize(block, n // 2)
        A = np.zeros((n, n))
        i = 2 * np.arange(n // 2)
        A[i, i], A[i + 1, i] = block, 1.0
        sgn = np.repeat(np.sign(block), 2) * np.tile([1.0, -1.0], n // 2)
        Ks = sp.csc_matrix((A[low], low), shape=(n, n))
        assert Ks.nnz == len(low[0])
        x, D, hits = clr.clr_ldl_solve(Ks, sgn, np.ones(n), order=np.arange(n), dyn_reg_eps=0.0)
        ref = -1.0 / block
        assert hits == 0 and np.array_equal(D[0::2], block)
        assert np.all(np.abs(D[1::2] - ref) <= np.spacing(np.abs(ref)))
