"""The triangular factor at the ends of the FP64 range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,h", [(1e-156, 0.3), (1e-120, 0.3), (1e120, 0.3), (1e151, 3.0)])
@pytest.mark.parametrize("n", [1, 5, 48, 130, 200])
def test_orthonormalisation_of_very_small_and_large_columns(scale, h, n):
    """Pivots down to 3e-310, whose reciprocal is no FP64 number, and up to 3e307, whose
    reciprocal is below the normal ones.  Tolerance: the smallest sums are multiples of 2^-1074, so at most some 1000
    partial sums and products are off by 2e-11 of a pivot together; n such terms."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(31, 31, 32, h)
    P = torch.from_numpy(np.random.default_rng(n).uniform(-1, 1, (g.npts, n)) * scale).cuda()
    api.orthonormalize(g, P)
    S = g.dV * (P.T @ P)
    assert (S - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max() <= (n + 8) * 2e-11
