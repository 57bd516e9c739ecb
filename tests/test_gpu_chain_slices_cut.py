"""Step (d) with its K cut into slices (tests/test_gemm_rules.py holds their numbers at these sizes): the last slice of 40
ranges, 8 more than the overlap and fewer than a flush interval (4,736 points), of whole intervals (4,096), of 48 after six
others (13,000), and several row tiles (23 orbitals).  4,608 points leave the last slice the overlap alone: not cut."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb,n_grid", [(12, 4096), (12, 4608), (12, 4736), (5, 13_000), (23, 6000)])
def test_sliced_assembly(n_orb, n_grid):
    from paper_2304_07006_gb300 import Context

    rng = np.random.default_rng(n_grid)
    dev = torch.device("cuda", 0)
    grid = torch.tensor(rng.normal(size=(n_grid, 3)) * 2.0, device=dev)
    w = torch.tensor(rng.uniform(0.5, 1.0, n_grid) / n_grid, device=dev)
    phi = torch.exp(-(grid ** 2).sum(1, keepdim=True) * 0.1) * torch.tensor(rng.normal(size=(n_grid, n_orb)), device=dev)
    gamma = torch.zeros(n_orb, n_orb, dtype=torch.float64, device=dev)
    gamma[0, 0] = gamma[1, 1] = 1.0
    terms = np.array([(0, 0, 1), (0, 1, 1), (1, 1, 1), (0, 1, 2)], dtype=np.int32)
    coef = rng.uniform(-0.1, 0.1, (1, 4))
    nuc = np.array([[0.0, 0.0, 0.7], [0.0, 0.0, -0.7]])

    def build(precision, chunks):
        """Delta U, as the sum over outer ranges of `chunks` points (small ones are not cut)."""
        total = torch.zeros((n_orb,) * 4, dtype=torch.float64, device=dev)
        with Context(precision) as ctx:
            ctx.set_jastrow(nuc, np.zeros(2, dtype=np.int32), terms, coef)
            for i in range(0, n_grid, chunks):
                ctx.set_outer_range(i, min(i + chunks, n_grid))
                dU = torch.empty((n_orb,) * 4, dtype=torch.float64, device=dev)
                dh = torch.empty(n_orb, n_orb, dtype=torch.float64, device=dev)
                ctx.build(grid, w, phi, gamma, dU=dU, dh=dh, e0=torch.empty(1, dtype=torch.float64, device=dev))
                total += dU
        return total

    cut, whole, exact = build("fp16x2", n_grid), build("fp16x2", 2048), build("fp64", n_grid)
    top = float(exact.abs().max())
    # FP32 intermediates (2^-24 each) and operands of 22 bits: 2e-6 of the largest entry; a lost range is 1e-3
    assert float((cut - exact).abs().max()) <= 2e-6 * top
    assert float((cut - whole).abs().max()) <= 2e-6 * top
