"""Setups through a user allocator (clr_set_allocator) that refuses: every failure is an
out-of-memory error of the call, and the next setup works."""
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
