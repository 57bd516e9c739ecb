"""Step (c) at the edges of its rank buckets (4, 8, 16 factors a pass) with more orbital rows than a round holds
(33 of 32): the oracle's Delta U."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rank", [1, 4, 5, 8, 9, 16, 17])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp16x2", 1e-6)])
def test_rank_buckets(precision, tol, rank):
    import synth
    from oracle import direct
    from paper_2304_07006_gb300 import Context

    p = synth.make_small(n_orb=33, n_rad=6, n_theta=3, n_phi=6, n_atoms=2, seed=11, n_occ=2)
    gamma = synth.random_density(p.n_orb, 3, rank=rank)
    ref = direct.build(p, gamma)
    with Context(precision) as ctx:
        ctx.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
        out = ctx.build(p.grid, p.weights, p.phi, gamma)
    # FP64 sums of about 200 points and 17 factors; FP32 intermediates and operands of 22 bits
    assert np.abs(out["dU"] - ref["dU"]).max() <= tol
