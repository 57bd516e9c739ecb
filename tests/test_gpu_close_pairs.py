"""F = lap_1 u + |grad_1 u|^2 of pairs of grid points that lie close together: H b'/r12 with H = du/db small or zero at
r12 = 0 (terms in b^2 only, or b terms far smaller than the b^2 ones) keeps its relative accuracy.

Tolerance 1e-13 of the largest entry: 2 H b'/r12 is within a few roundings (2^-53) of itself on either side, and its pairs
are no larger in the sums than the others."""
import numpy as np
import pytest

import synth
from oracle import two_body_k

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("terms,coef", [
    ([(0, 0, 2)], [0.07]),                                    # H = 0 at r12 = 0
    ([(0, 0, 2), (1, 1, 2)], [0.07, -0.09]),
    ([(0, 0, 1), (0, 1, 2), (1, 2, 1)], [1e-9, 0.08, -2e-9]), # H far smaller there than elsewhere
    ([(0, 0, 1), (0, 0, 2), (0, 1, 1), (1, 1, 0)], [0.0, 0.1, 0.0, 0.05]),
])
@pytest.mark.parametrize("dist", [1e-3, 1e-7, 1e-11, 5e-15])   # the last: coincident
def test_close_pairs(terms, coef, dist):
    terms = np.array(terms, dtype=np.int32)
    p = synth.make_small(n_orb=5, n_rad=5, n_theta=4, n_phi=5, n_atoms=2, seed=21, terms=terms)   # 200 points
    p.coef = np.stack([np.array(coef), 1.5 * np.array(coef)])
    dphi = synth.orbital_gradients(p)
    for k in (20, 60, 100):      # the x coordinates of the partners are zero, so that the distances are exact
        p.grid[k, 0] = 0.0
        p.grid[k + 1] = p.grid[k] + np.array([dist, 0.0, 0.0])
    want = two_body_k.k_integrals(p.grid, p.weights, p.phi, dphi, p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    from paper_2304_07006_gb300 import Context
    with Context("fp64") as c:
        c.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
        got = c.two_body_K(p.grid, p.weights, p.phi, dphi)
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
