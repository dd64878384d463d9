"""The symbolic factorization and the scaling of a cohort through the binding (no GPU)."""
import numpy as np

from paper_2412_19027_gb300 import build, clr, workloads as W


def setup_module():
    build.build()


def test_symbolic_and_scaling_cover_the_whole_cohort():
    """Both describe the merged problem: arrays of all problems' variables and rows, the later ones larger than
    the first."""
    probs = [W.nonneg_qp(k, n=10 + 7 * k, m=20 + 13 * k) for k in range(4)]
    args = [(p.P, p.q, p.A, p.b, p.cones) for p in probs]
    n, m = sum(len(p.q) for p in probs), sum(len(p.b) for p in probs)
    many = clr.clr_batch_analyze(args)
    sym = many.symbolic()
    assert sorted(sym["row_perm"]) == list(range(m)) and sorted(sym["perm"]) == list(range(n + m))
    D, E, _ = many.scaling()
    assert D.shape == (n,) and E.shape == (m,) and np.all(D > 0) and np.all(E > 0)
    one = clr.clr_analyze(*args[0])
    assert one.symbolic()["row_perm"].shape == (20,) and one.scaling()[0].shape == (10,)
