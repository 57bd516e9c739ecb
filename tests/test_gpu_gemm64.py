"""The FP64 path on the tensor cores (digit planes, grad64.cu and gemm64_tc.cu) at the edges of its tiles and
blocks: odd sizes around the 128 x 32 tiles and 64-wide ranges, more nuclei than the mixed precisions take,
blocks of inner points, outer points and step (d) values (XTC_D64_BUDGET scales their memory budgets),
points on nuclei and coincident points.

Tolerance 1e-13 of the largest entry of each output: both sides sum K <= 4,096 FP64 terms, an FP64 sum of K
random-sign terms errs by about sqrt(K) 2^-53 = 7e-15 of the operand norms, the digits by 2^-71 of the row
maxima per term."""
import numpy as np
import pytest

import synth
from oracle import direct, two_body_k

pytestmark = pytest.mark.gpu

TOL = 1e-13


def _ctx(p):
    from paper_2304_07006_gb300 import Context
    c = Context("fp64")
    c.set_jastrow(p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    return c


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


@pytest.mark.parametrize("budget", [None, "1e-6"])
@pytest.mark.parametrize("n_orb,n_rad,n_theta,n_phi,n_atoms", [
    (2, 2, 2, 3, 1),     # 12 points, three pairs (with one orbital Delta U vanishes identically)
    (7, 4, 4, 4, 2),     # 128 points, 28 pairs (inside one column tile)
    (8, 5, 5, 5, 2),     # 250 points, 36 pairs (a ragged second column tile)
    (11, 7, 5, 5, 3),    # 525 points, 66 pairs
])
def test_fp64_build_at_the_edges(monkeypatch, budget, n_orb, n_rad, n_theta, n_phi, n_atoms):
    if budget:
        monkeypatch.setenv("XTC_D64_BUDGET", budget)   # blocks of 128 inner and outer points
    p = synth.make_small(n_orb=n_orb, n_rad=n_rad, n_theta=n_theta, n_phi=n_phi, n_atoms=n_atoms, seed=17)
    p.grid[1] = p.nuc_xyz[0]          # a point on a nucleus
    if p.n_grid > 20:
        p.grid[9] = p.grid[4]         # coincident points
    g = synth.random_density(n_orb, 2)
    ref = direct.build(p, g)
    with _ctx(p) as c:
        out = c.build(p.grid, p.weights, p.phi, g)
        c.set_outer_range(3, min(140, p.n_grid))
        part = c.build(p.grid, p.weights, p.phi, g)
    assert _rel(out["dU"], ref["dU"]) < TOL
    want = direct.build(p, g, outer=np.arange(3, min(140, p.n_grid)))
    assert _rel(part["dU"], want["dU"]) < TOL and _rel(part["dh"], want["dh"]) < TOL


def test_fp64_vfield_with_more_nuclei_than_the_mixed_path_takes():
    p = synth.make_small(n_orb=5, n_rad=5, n_theta=4, n_phi=5, n_atoms=4, seed=3)
    rng = np.random.default_rng(0)
    p.nuc_xyz = np.concatenate([p.nuc_xyz, rng.uniform(-2, 2, (7, 3))])
    p.nuc_set = np.concatenate([p.nuc_set, np.arange(7, dtype=np.int32) % p.n_sets]).astype(np.int32)
    from paper_2304_07006_gb300 import unpack_pairs
    want = direct.vfield(p.grid, p.weights, p.phi, (p.nuc_xyz, p.nuc_set, p.terms, p.coef), np.arange(5, 205))
    with _ctx(p) as c:
        got = unpack_pairs(c.vfield(p.grid, p.weights, p.phi, 5, 205), p.n_orb)
    assert _rel(got, want) < TOL


@pytest.mark.parametrize("budget", [None, "1e-6"])
def test_k_in_blocks_with_coincident_points(monkeypatch, budget):
    if budget:
        monkeypatch.setenv("XTC_D64_BUDGET", budget)
    p = synth.make_small(n_orb=7, n_rad=6, n_theta=5, n_phi=5, n_atoms=2, seed=8)   # 300 points
    p.grid[0], p.grid[5] = p.nuc_xyz[1], p.grid[6]
    dphi = synth.orbital_gradients(p)
    want = two_body_k.k_integrals(p.grid, p.weights, p.phi, dphi, p.nuc_xyz, p.nuc_set, p.terms, p.coef)
    with _ctx(p) as c:
        got = c.two_body_K(p.grid, p.weights, p.phi, dphi)
    assert _rel(got, want) < TOL


def test_rows_of_very_different_magnitude():
    """Digits are relative to each row's maximum: scaled orbitals scale the results exactly."""
    p = synth.make_small(n_orb=4, n_rad=5, n_theta=4, n_phi=4, n_atoms=2, seed=4)
    s = 2.0 ** np.array([0, 300, -300, 40])
    with _ctx(p) as c:
        V = c.vfield(p.grid, p.weights, p.phi, 0, p.n_grid)
        Vs = c.vfield(p.grid, p.weights, p.phi * s, 0, p.n_grid)
    i, j = np.triu_indices(4)
    assert np.array_equal(Vs, V * (s[i] * s[j]))
