"""The row kernels of the learned preconditioner on grids above the sizes that go
a thread to a point, with rows that end inside a group of four lattice positions,
against a plain FP64 evaluation of some of the columns, at both sides of each size rule.
Tolerance: as for the small grids (test_net_edges_gpu).
"""
import numpy as np
import pytest

import workloads as wl
from tests.test_net_edges_gpu import _net

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,nb", [((19, 21, 25), 16), ((22, 21, 23), 16), ((22, 21, 23), 33), ((25, 26, 27), 4), ((27, 26, 26), 4),
                                    ((26, 26, 27), 12), ((27, 26, 26), 15), ((31, 31, 32), 8), ((33, 31, 31), 8),
                                    ((35, 37, 38), 6), ((37, 37, 37), 10), ((53, 54, 53), 5), ((54, 53, 53), 7)])
def test_net_rows(box, nb):
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(*box, 0.3, order=1)           # lexicographic: points in box order
    H = api.Hamiltonian(g, np.zeros(g.npts))
    R = torch.from_numpy(np.random.default_rng(nb).uniform(-1, 1, (g.npts, nb)).astype(np.float32)).cuda()
    ws = wl.conv_init(3)
    w = torch.from_numpy(np.concatenate([a.reshape(-1) for a in ws])).cuda()
    got = api.precond_apply(H, w, R).double().cpu().numpy()
    wq = [torch.from_numpy(a).to(torch.bfloat16).double().numpy() for a in ws]
    r = R.cpu().numpy()
    assert np.isfinite(got).all()
    for k in {0, nb // 2, nb - 1}:
        rms = np.sqrt(np.mean(r[:, k].astype(np.float64) ** 2))
        x = torch.from_numpy(r[:, k] * np.float32(1.0 / rms)).to(torch.bfloat16).double().numpy()
        ref = rms * _net(box, x, wq, True)
        mag = rms * _net(box, np.abs(x), [np.abs(a) for a in wq], False)
        assert np.all(np.abs(got[:, k] - ref) <= 3 * 216 * 2.0 ** -23 * mag)
