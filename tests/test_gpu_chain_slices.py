"""Step (d) with its K cut into slices (few orbital pairs): the FP64 path's Delta U, where the last slice is as short as it may
be (2,688 points: 128 + 40 ranges), one range group too short to be cut off (2,560), and at uneven lengths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb,n_grid", [(12, 2560), (12, 2688), (5, 4100), (23, 6000)])
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
    out = {}
    for precision in ("fp64", "fp16x2"):
        with Context(precision) as ctx:
            ctx.set_jastrow(np.array([[0.0, 0.0, 0.7], [0.0, 0.0, -0.7]]), np.zeros(2, dtype=np.int32), terms, coef)
            dU = torch.empty((n_orb,) * 4, dtype=torch.float64, device=dev)
            dh, e0 = torch.empty(n_orb, n_orb, dtype=torch.float64, device=dev), torch.empty(1, dtype=torch.float64, device=dev)
            ctx.build(grid, w, phi, gamma, dU=dU, dh=dh, e0=e0)
            out[precision] = dU
    # FP32 intermediates (2^-24 each) and operands of 22 bits: 2e-6 of the largest entry; a lost range is 1e-3
    assert float((out["fp16x2"] - out["fp64"]).abs().max()) <= 2e-6 * float(out["fp64"].abs().max())
