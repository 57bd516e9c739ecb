"""FP64 contractions with grid points where the density leaves the normal FP64 range (far points of tight orbitals): their
pair products are subnormal or zero, contribute nothing, and leave the other points' accuracy alone.

Tolerance 1e-13 of the largest entry: sums of a few hundred FP64 terms, as in the other tests of these contractions."""
import numpy as np
import pytest

import synth
from oracle import direct, two_body_k

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponents", [(-505,), (-512,), (-518, -525), (-531, -535, -537), (-600,), (-1060,)])
def test_points_of_subnormal_density(exponents):
    from paper_2304_07006_gb300 import Context, unpack_pairs
    p = synth.make_small(n_orb=5, n_rad=5, n_theta=5, n_phi=5, n_atoms=2, seed=30)   # 250 points
    dphi = synth.orbital_gradients(p)
    rng = np.random.default_rng(1)
    for k, e in enumerate(exponents):
        for row in (7 + 40 * k, 130 + k):
            p.weights[row] = 1.0
            p.phi[row] = rng.uniform(0.5, 1.0, p.n_orb) * 2.0 ** e
            dphi[row] = rng.uniform(0.5, 1.0, (p.n_orb, 3)) * 2.0 ** e
    g = synth.random_density(p.n_orb, 2)
    jas = (p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    want = direct.build(p, g)
    with Context("fp64") as c:
        c.set_jastrow(*jas)
        V = unpack_pairs(c.vfield(p.grid, p.weights, p.phi, 0, p.n_grid), p.n_orb)
        out = c.build(p.grid, p.weights, p.phi, g)
        K = c.two_body_K(p.grid, p.weights, p.phi, dphi)
    for got, ref in ((V, direct.vfield(p.grid, p.weights, p.phi, jas, np.arange(p.n_grid))),
                     (out["dU"], want["dU"]), (out["dh"], want["dh"]),
                     (K, two_body_k.k_integrals(p.grid, p.weights, p.phi, dphi, *jas))):
        assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()
