"""The Hartree solver's transforms at axis lengths of every radix (powers of
two, powers of three, both), odd and even numbers of lines, and a single
point, against numpy's FFT of the same cube and kernel.

Tolerance: a transform of n points is off by at most about 4 u log2(n) of its
2-norm; forward and inverse transform and the kernel give 8 u log2(n) + 2 u
of the 2-norm of the potential on the whole cube, on both sides.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,h", [((1, 1, 1), 0.3), ((2, 3, 5), 0.4), ((7, 4, 9), 0.3), ((11, 11, 3), 0.5), ((16, 8, 3), 0.3),
                                   ((20, 33, 11), 0.25), ((5, 40, 12), 0.3), ((3, 2, 60), 0.3)])
def test_poisson_sizes(box, h):
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(*box, h)
    P = api.Poisson(g)
    N, rc, _ = P.info()
    n = np.random.default_rng(sum(box)).uniform(-1, 1, g.npts)
    u = g.ijk()
    u = u - u.min(0)
    cube = np.zeros(N)
    cube[u[:, 0], u[:, 1], u[:, 2]] = n
    f = [2 * np.pi * np.fft.fftfreq(k, d=h) for k in N]
    G2 = f[0][:, None, None] ** 2 + f[1][None, :, None] ** 2 + f[2][None, None, :] ** 2
    G2[0, 0, 0] = 1.0
    vg = 4 * np.pi * (1 - np.cos(np.sqrt(G2) * rc)) / G2
    vg[0, 0, 0] = 2 * np.pi * rc * rc
    full = np.fft.ifftn(np.fft.fftn(cube) * vg).real
    dev = torch.from_numpy(n).cuda()
    V = P.solve(dev).cpu().numpy()
    eps = 2.0 ** -53
    err = V - full[u[:, 0], u[:, 1], u[:, 2]]
    assert np.linalg.norm(err) <= 2 * (8 * np.log2(full.size) + 2) * eps * np.linalg.norm(full)
    # a second solve on the same plan starts from a clean box
    assert np.array_equal(P.solve(dev).cpu().numpy(), V)
