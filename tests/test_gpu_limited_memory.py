"""FP64 calls and K where little device memory is left: the blocks of digits shrink until they fit, and a call is refused
only when 128-point blocks do not fit either.  A caller allocator with a limit on its total stands in for the GPU's memory."""
import numpy as np
import pytest

import synth
from oracle import direct, two_body_k

pytestmark = pytest.mark.gpu


class _Allocator:
    def __init__(self, limit):
        self.limit, self.live, self.peak = limit, {}, 0

    def total(self):
        return sum(t.numel() for t in self.live.values())

    def alloc(self, n):
        import torch
        if self.total() + n > self.limit:
            return 0
        t = torch.empty(n, dtype=torch.uint8, device="cuda:0")
        self.live[t.data_ptr()] = t
        self.peak = max(self.peak, self.total())
        return t.data_ptr()

    def release(self, ptr):
        del self.live[ptr]


# 4,000 points, 12 orbitals: rho^T in FP64 is 2.5 MB, the digits of all pair functions at once 0.8 GB
LIMIT = 200 << 20


@pytest.fixture(scope="module")
def problem():
    p = synth.make_small(n_orb=12, n_rad=20, n_theta=10, n_phi=10, n_atoms=2, seed=3, n_occ=2)
    return p, synth.orbital_gradients(p)


def _ctx(p, prec, a=None):
    from paper_2304_07006_gb300 import Context
    c = Context(prec, **({"allocator": (a.alloc, a.release)} if a else {}))
    c.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    return c


def test_fp64_calls_fit_little_memory(problem):
    p, dphi = problem
    gb = synth.random_density(p.n_orb, 5, rank=2)
    calls = {
        "build": lambda c: c.build(p.grid, p.weights, p.phi, p.gamma)["dU"],
        "rohf": lambda c: c.build_rohf(p.grid, p.weights, p.phi, p.gamma, gb)["dU_ab"],
        "vfield": lambda c: c.vfield(p.grid, p.weights, p.phi, 0, p.n_grid),
        "K": lambda c: c.two_body_K(p.grid, p.weights, p.phi, dphi),
    }
    for name, call in calls.items():
        with _ctx(p, "fp64") as c:
            want = call(c)
        a = _Allocator(LIMIT)
        with _ctx(p, "fp64", a) as c:
            got, again = call(c), call(c)
        assert not a.live
        # blocks change the order of FP64 additions only
        assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max(), name
        assert np.array_equal(got, again), name


def test_memory_too_small_for_any_block_is_refused(problem):
    from paper_2304_07006_gb300 import XtcError
    p, _ = problem
    a = _Allocator(2 << 20)
    with _ctx(p, "fp64", a) as c:
        with pytest.raises(XtcError) as e:
            c.build(p.grid, p.weights, p.phi, p.gamma)
        assert e.value.code == -4
        # and the context still builds what fits
        a.limit = LIMIT
        out = c.build(p.grid, p.weights, p.phi, p.gamma)
    with _ctx(p, "fp64") as c:
        want = c.build(p.grid, p.weights, p.phi, p.gamma)
    assert np.abs(out["dU"] - want["dU"]).max() <= 1e-14 * np.abs(want["dU"]).max()


@pytest.mark.parametrize("text", ["nan", "inf", "-1", "0", "1e300", "junk", ""])
def test_a_budget_scale_that_is_none_leaves_the_default(monkeypatch, problem, text):
    p, _ = problem
    peaks = []
    for value in (None, text):
        if value is not None:
            monkeypatch.setenv("XTC_D64_BUDGET", value)
        a = _Allocator(8 << 30)
        with _ctx(p, "fp64", a) as c:
            c.vfield(p.grid, p.weights, p.phi, 0, 256)
        peaks.append(a.peak)
    assert peaks[0] == peaks[1]
