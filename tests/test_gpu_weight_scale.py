"""FP64 results scale with the weights: every contraction's operands carry scales that move with them, so powers of 2 on the
weights leave all digits alone, and the results are the same numbers with other exponents (Delta U, Delta h and e0 with the
cube, K with the square)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-120, -40, 60])
def test_weights_scaled_by_powers_of_two(power):
    from paper_2304_07006_gb300 import Context
    p = synth.make_small(n_orb=6, n_rad=6, n_theta=5, n_phi=5, n_atoms=2, seed=31)   # 300 points
    dphi = synth.orbital_gradients(p)
    g, gb = synth.random_density(p.n_orb, 2), synth.random_density(p.n_orb, 3, rank=2)
    out = {}
    for s in (0, power):
        w = p.weights * 2.0 ** s
        with Context("fp64") as c:
            c.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
            a = c.build(p.grid, w, p.phi, g)
            b = c.build_rohf(p.grid, w, p.phi, g, gb)
            out[s] = {"dU": a["dU"], "dh": a["dh"], "e0": a["e0"], "ab": b["dU_ab"], "dh_b": b["dh_b"],
                      "K": c.two_body_K(p.grid, w, p.phi, dphi)}
    for k, want in out[0].items():
        assert np.array_equal(out[power][k], np.asarray(want) * 2.0 ** ((2 if k == "K" else 3) * power)), k
