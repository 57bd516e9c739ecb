"""A GEMM of many waves runs as several launches: its rows are those of a GEMM that fits one launch, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16x2", "bf16x3"])
def test_rows_do_not_depend_on_the_launch(precision):
    from paper_2304_07006_gb300 import Context

    n_grid, n_orb = 20000, 40            # 3,304 and 2,826 CTAs, 1,520 a launch
    rng = np.random.default_rng(5)
    dev = torch.device("cuda", 0)
    grid = torch.tensor(rng.normal(size=(n_grid, 3)) * 2.0, device=dev)
    w = torch.tensor(rng.uniform(0.01, 1.0, n_grid), device=dev)
    phi = torch.exp(-(grid ** 2).sum(1, keepdim=True) * 0.2) * torch.tensor(rng.normal(size=(n_grid, n_orb)), device=dev)
    n_pair = n_orb * (n_orb + 1) // 2
    terms = np.array([(0, 0, 1), (0, 1, 1), (1, 1, 1), (0, 1, 2)], dtype=np.int32)

    def field(begin, end):
        out = torch.empty(end - begin, 3, n_pair, dtype=torch.float64, device=dev)
        ctx.vfield(grid, w, phi, begin, end, out=out)
        return out

    with Context(precision) as ctx:
        ctx.set_jastrow(np.array([[0.0, 0.0, 0.7], [0.0, 0.0, -0.7]]), np.zeros(2, dtype=np.int32), terms,
                        rng.uniform(-0.1, 0.1, (1, 4)))
        whole = field(0, n_grid)
        for begin, end in ((0, 100), (9984, 10240), (19900, 20000)):
            assert torch.equal(whole[begin:end], field(begin, end))
        assert float(whole.abs().max()) > 0
