"""Setups through a user allocator (clr_set_allocator) with little room: what setup needs gives an
out-of-memory error, what it can do without is left out, and the next setup works."""
import ctypes as C

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


class Budget:
    """A user allocator over at most `limit` bytes, its `refuse`-th call refused, by torch's allocator."""

    def __init__(self, limit, refuse=None):
        self.limit, self.refuse, self.used, self.peak, self.calls, self.held = limit, refuse, 0, 0, 0, {}
        fa, ff = C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p), C.CFUNCTYPE(None, C.c_void_p, C.c_size_t, C.c_void_p)
        self.fns = fa(self.alloc), ff(self.free)

    def alloc(self, n, ctx):
        self.calls += 1
        if self.used + n > self.limit or self.calls == self.refuse:
            return None
        self.used += n
        self.peak = max(self.peak, self.used)
        t = torch.empty(n, dtype=torch.uint8, device="cuda")
        self.held[t.data_ptr()] = t
        return t.data_ptr()

    def free(self, p, n, ctx):
        self.used -= n
        del self.held[p]

    def __enter__(self):
        L = clr._lib()
        L.clr_set_allocator.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p]
        assert L.clr_set_allocator(C.cast(self.fns[0], C.c_void_p), C.cast(self.fns[1], C.c_void_p), None) == 0
        return self

    def __exit__(self, *a):
        assert not self.held
        clr._lib().clr_set_allocator(None, None, None)


OOM = -4  # CLR_E_OOM


# every allocation of a setup refused in turn: the error, never a null buffer in a kernel
@pytest.mark.parametrize("bits", [64, 32])
def test_each_refused_allocation_is_reported(bits):
    p = W.mixed_cone(1, n=60, n_zero=10, n_nonneg=90, n_soc=10, n_exp=3, n_pow=3)
    arg = (p.P, p.q, p.A, p.b, p.cones, clr.clr_default_settings(bits, max_iter=3, fp64_escalation=0))
    with Budget(1 << 40) as m:
        sv = clr.clr_setup(*arg)
        total = m.calls
        sv.free()
    assert total > 50
    for k in range(1, total + 1):
        with Budget(1 << 40, refuse=k) as m:
            with pytest.raises(clr.ClrError) as e:
                clr.clr_setup(*arg)
            assert e.value.code == OOM, (k, e.value)
    sv = clr.clr_setup(*arg)
    sv.solve()
    assert np.all(np.isfinite(sv.solution()[0]))
    sv.free()


def test_refused_allocations_of_the_cone_steps():
    rng = np.random.default_rng(0)
    cones = [(W.NONNEG, 5, 0.0), (W.SOC, 4, 0.0)]
    s = np.r_[1.0 + rng.random(5), 3.0, rng.standard_normal(3)]
    with Budget(1 << 40) as m:
        ref = clr.clr_cones_step_length(cones, s, s, -s, -s, 1e6)
        total = m.calls
    for k in range(1, total + 1):
        with Budget(1 << 40, refuse=k):
            with pytest.raises(clr.ClrError) as e:
                clr.clr_cones_step_length(cones, s, s, -s, -s, 1e6)
            assert e.value.code == OOM
    assert clr.clr_cones_step_length(cones, s, s, -s, -s, 1e6) == ref


def dense_qp(seed, n):
    """A QP whose KKT factorization has a root of about n rows."""
    import scipy.sparse as sp
    rng = np.random.default_rng(seed)
    H = rng.standard_normal((n, n)) / np.sqrt(n)
    A = sp.csc_matrix(sp.vstack([sp.eye(n), -sp.eye(n)]))
    return (sp.csc_matrix(np.triu(H @ H.T + 0.1 * np.eye(n))), rng.standard_normal(n), A, np.ones(2 * n),
            [(W.NONNEG, 2 * n, 0.0)])


def solve_in(limit, probs, schedule):
    """(solutions, routes, largest use) of a cohort set up and solved in `limit` bytes."""
    st = clr.clr_default_settings(64, max_iter=5, big_front_schedule=schedule)
    with Budget(limit) as m:
        sv = clr.clr_batch_setup(probs, st)
        sv.solve()
        out = [sv.solution_of(i) for i in range(len(probs))], sv.routes(), m.peak
        sv.free()
        assert m.used == 0
    return out


def same(a, b):
    for u, v in zip(a, b):
        for x, y in zip(u[:3], v[:3]):
            np.testing.assert_array_equal(x, y)


# The scratch of the digit products is what setup can do without: where everything else fits, setup is
# not refused.  First no room for it (FMA products, the bits of schedule 2), then room for one front's
# at a time (the bits of all of them at once).
def test_digit_scratch_within_a_memory_limit():
    probs = [dense_qp(k, 400 + 7 * k) for k in range(3)]
    fma, r2, least = solve_in(1 << 40, probs, 2)
    full, r1, most = solve_in(1 << 40, probs, 1)
    assert r2["digit_fronts"] == 0 and r1["digit_fronts"] == 3 and r1["digit_launches"] == 1
    front = r1["digit_bytes"] / 3  # about that of each
    slack = 1 << 20  # task tables of both kinds, less than a front's scratch
    assert front > 2 * slack and most - least > 3 * front - slack
    got, r, peak = solve_in(least + slack, probs, 1)
    assert r["digit_no_room"] == 1 and r["digit_fronts"] == 0
    same(got, fma)
    got, r, peak = solve_in(least + slack + int(1.2 * front), probs, 1)
    assert r["digit_no_room"] == 0 and r["digit_fronts"] == 3 and r["digit_launches"] == 3
    same(got, full)


# a problem's products are chosen by its own fronts: the same alone and in a cohort
def test_digits_alone_and_in_a_cohort():
    probs = [dense_qp(10 + k, n) for k, n in enumerate((330, 400, 470))]
    both, _, _ = solve_in(1 << 40, probs, 1)
    for p, b in zip(probs, both):
        one, r, _ = solve_in(1 << 40, [p], 1)
        assert r["digit_fronts"] == 1
        same(one, [b])
