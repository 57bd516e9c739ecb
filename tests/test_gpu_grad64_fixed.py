"""The FP64 pair fields with Jastrow coefficients of very different magnitudes (the fixed-point scales of an outer
point), terms without a part in one electron, a point on a nucleus, coincident and far points: against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("terms", [
    [(0, 0, 1), (0, 1, 1), (1, 2, 1), (1, 1, 2)],      # the usual mixture
    [(1, 1, 0), (2, 2, 2)],                            # nothing left where a = 0
    [(0, 0, 2)],                                       # no nuclear terms
])
@pytest.mark.parametrize("scale", [(1.0, 1.0), (1e-7, 1e3), (1e12, 0.0)])
def test_fixed_point_scales(terms, scale):
    from oracle import jastrow
    from paper_2304_07006_gb300 import Context

    rng = np.random.default_rng(len(terms))
    n_grid, n_orb = 200, 2
    nuc = np.array([[0.0, 0.0, -0.7], [0.0, 0.3, 0.9], [1.5, 0.0, 0.0]])
    sets = np.array([0, 1, 1], dtype=np.int32)
    terms = np.array(terms, dtype=np.int32)
    coef = rng.uniform(-0.1, 0.1, (2, len(terms))) * np.array(scale)[:, None]
    grid = rng.normal(size=(n_grid, 3)) * 2.0
    grid[3], grid[7], grid[8] = nuc[0], grid[6], [300.0, -200.0, 50.0]
    w = rng.uniform(0.1, 1.0, n_grid)
    phi = rng.normal(size=(n_grid, n_orb))
    with Context("fp64") as ctx:
        ctx.set_jastrow(nuc, sets, terms, coef)
        V = ctx.vfield(grid, w, phi, 0, n_grid)
    G = jastrow.grad1(grid[:, None, :], grid[None, :, :], nuc, sets, terms, coef)
    rho = np.stack([w * phi[:, p] * phi[:, q] for p, q in ((0, 0), (0, 1), (1, 1))])
    ref = np.einsum("ijx,kj->ixk", G, rho)
    # sums of 200 FP64 terms, each within a few roundings of the largest partial term: 1e-13 of the largest entry
    assert np.abs(V.reshape(ref.shape) - ref).max() <= 1e-13 * np.abs(ref).max()
