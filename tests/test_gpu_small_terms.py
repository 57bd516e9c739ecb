"""FP64 pair fields whose terms vanish where the weight is: both electrons of every term within a small distance of one
nucleus, or of each other, where a2 and b are small and no term is left at a2 = 0.  The fixed-point evaluation of an outer
point's row resolves 2^-59 of the sum of its coefficients, so such rows are evaluated in FP64 instead.

Tolerance 1e-13 of the largest entry: FP64 sums of 300 terms, rows that stand 2^46 above the fixed point's unit."""
import numpy as np
import pytest

from oracle import jastrow, two_body_k

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("terms", [[(1, 2, 1), (2, 2, 1)], [(1, 1, 2)], [(2, 2, 0), (1, 1, 1)], [(0, 0, 1), (1, 2, 2)]])
@pytest.mark.parametrize("length", [1.0, 1e-4, 1e-9])
@pytest.mark.parametrize("spread", [False, True])
def test_small_terms(terms, length, spread):
    from paper_2304_07006_gb300 import Context
    rng = np.random.default_rng(8)
    n, N = 300, 3
    terms = np.array(terms, dtype=np.int32)
    nuc, sets, coef = np.zeros((1, 3)), np.zeros(1, dtype=np.int32), rng.uniform(-0.1, 0.1, (1, len(terms)))
    grid = rng.normal(size=(n, 3)) * length
    w = rng.uniform(0.1, 1.0, n)
    phi = rng.normal(size=(n, N))
    if spread:                       # outer points of ordinary distance, without density
        grid[::3] = rng.normal(size=(len(grid[::3]), 3)) * 2.0
        phi[::3] *= 1e-30
    dphi = rng.normal(size=(n, N, 3)) / length
    with Context("fp64") as c:
        c.set_jastrow(nuc, sets, terms, coef)
        V = c.vfield(grid, w, phi, 0, n)
        K = c.two_body_K(grid, w, phi, dphi)
    G = jastrow.grad1(grid[:, None, :], grid[None, :, :], nuc, sets, terms, coef)
    i, j = np.triu_indices(N)
    want = np.einsum("ijx,jk->ixk", G, w[:, None] * phi[:, i] * phi[:, j])
    err, top = np.abs(V.reshape(want.shape) - want).max(axis=(1, 2)), np.abs(want).max(axis=(1, 2))
    assert (err <= 1e-13 * top).all()
    ref = two_body_k.k_integrals(grid, w, phi, dphi, nuc, sets, terms, coef)
    assert np.abs(K - ref).max() <= 1e-13 * np.abs(ref).max()
