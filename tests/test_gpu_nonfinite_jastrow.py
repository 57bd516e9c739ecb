"""Finite Jastrow coefficients whose sums leave the FP64 range: the pair fields are infinities or NaN, never numbers."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("term", [(0, 0, 1), (1, 1, 0), (1, 1, 2)])
def test_overflowing_coefficients_are_not_numbers(term):
    from paper_2304_07006_gb300 import Context
    terms = np.array([term, (0, 0, 1)], dtype=np.int32)
    p = synth.make_small(n_orb=3, n_rad=4, n_theta=3, n_phi=4, n_atoms=2, seed=6, terms=terms)
    p.coef = np.full((2, 2), 1.0)
    p.coef[:, 0] = 1.7e308
    p.grid = p.grid + np.array([0.3, 0.0, 0.0])   # no point on a nucleus
    with Context("fp64") as c:
        c.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
        V = c.vfield(p.grid, p.weights, p.phi, 0, p.n_grid)
        K = c.two_body_K(p.grid, p.weights, p.phi, synth.orbital_gradients(p))
    assert not np.isfinite(V).any(axis=(1, 2)).all()
    assert not np.isfinite(K).all()
