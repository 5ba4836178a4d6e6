"""Blocks whose rows lie 4 GB or more apart (a few rows of a very wide array)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("extra", [0, 64])
def test_overlap_of_far_rows(dtype, extra):
    """Tolerance: three products and sums in FP64."""
    from paper_1306_2953_gb300 import api
    t, es = (torch.float64, 8) if dtype == "f64" else (torch.float32, 4)
    ld, n = 2 ** 32 // es + extra, 40
    g = api.Grid.box(3, 1, 1, 0.3)
    buf = torch.empty(2 * ld + n, dtype=t, device="cuda")
    X = buf.as_strided((3, n), (ld, 1))
    X.copy_(torch.from_numpy(np.random.default_rng(1).uniform(-1, 1, (3, n))).to(t))
    Y = torch.from_numpy(np.random.default_rng(2).uniform(-1, 1, (3, 7))).to(t).cuda()
    x, y = X.double(), Y.double()
    for A, B, a, b in ((X, Y, x, y), (Y, X, y, x), (X, X, x, x)):
        err = (api.overlap(g, A, B) - g.dV * (a.T @ b)).abs()
        assert bool((err <= 8 * 2.0 ** -53 * g.dV * (a.abs().T @ b.abs())).all())
