"""Two-body integrals K with an outer point next to a nucleus and a weight to match: W grows as 1/r there, the point itself
contributes nothing, and every other point keeps its accuracy.

Tolerance 1e-13 of the largest entry, as for the other FP64 contractions of K <= 4,096 terms: sqrt(K) 2^-53 = 7e-15 from
either side's sums, digits 2^-71 of a row's maximum."""
import numpy as np
import pytest

import synth
from oracle import two_body_k

pytestmark = pytest.mark.gpu

TOL = 1e-13


def _k(p, dphi):
    from paper_2304_07006_gb300 import Context
    with Context("fp64") as c:
        c.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
        return c.two_body_K(p.grid, p.weights, p.phi, dphi)


@pytest.mark.parametrize("n_orb,dist,weight", [
    (6, 1e-8, 1e-24),
    (6, 1e-10, 1e-30),
    (7, 1e-12, 1e-36),     # a weight of r^3
    (7, 1e-12, -1e-36),
    (6, 2e-14, 0.0),
])
def test_point_next_to_a_nucleus(n_orb, dist, weight):
    p = synth.make_small(n_orb=n_orb, n_rad=5, n_theta=5, n_phi=8, n_atoms=2, seed=12)   # 400 points
    dphi = synth.orbital_gradients(p)
    p.grid[11] = p.nuc_xyz[1] + np.array([dist, 0.0, 0.0])   # the nucleus is at x = 0
    p.weights[11] = weight
    want = two_body_k.k_integrals(p.grid, p.weights, p.phi, dphi, p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    assert np.abs(_k(p, dphi) - want).max() <= TOL * np.abs(want).max()


def test_scaled_orbitals_scale_k_exactly():
    """The point scales are taken from every orbital at one height: powers of 2 on the orbitals leave the digits alone."""
    p = synth.make_small(n_orb=4, n_rad=5, n_theta=4, n_phi=4, n_atoms=2, seed=4)
    p.weights[3] = 0.0
    p.phi[7] = 0.0            # a point without density, gradients left
    dphi = synth.orbital_gradients(p)
    s = 2.0 ** np.array([0, 100, -100, 30])
    K, Ks = _k(p, dphi), None
    p.phi = p.phi * s
    Ks = _k(p, dphi * s[:, None])
    assert np.array_equal(Ks, K * np.einsum("p,q,r,s->pqrs", s, s, s, s))


@pytest.mark.parametrize("length", [1e-12, 1e-6, 1e6])
def test_grids_of_other_lengths(length):
    """W and the gradients have a length in them, V and the orbitals do not: neither part of an operand row takes bits from the
    other, whatever their sizes."""
    rng = np.random.default_rng(5)
    p = synth.make_small(n_orb=5, n_rad=5, n_theta=4, n_phi=5, n_atoms=1, seed=14)   # 100 points around one nucleus
    p.nuc_xyz = np.zeros((1, 3))
    p.grid = rng.normal(size=p.grid.shape) * length
    dphi = rng.normal(size=(p.n_grid, p.n_orb, 3)) * np.abs(p.phi).max() / length
    want = two_body_k.k_integrals(p.grid, p.weights, p.phi, dphi, p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    assert np.abs(_k(p, dphi) - want).max() <= TOL * np.abs(want).max()
