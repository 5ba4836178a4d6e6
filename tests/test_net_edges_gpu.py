"""The network on the grid at every kind of column count (a tensor-core tile
holds 16 states), on grids whose rows end inside a group of four lattice
positions, and with strided blocks, against a plain FP64 evaluation.

Tolerance: activations are exact in their pieces; each of the three layers adds
at most 216 FP32 roundings or truncations of its magnitude sums, bounded by
216 * 2^-23 of the network evaluated with absolute values, times three.
"""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _net(box, x, ws, relu):
    """x [points], box (n0, n1, n2) full box, ws three [co, ci, 3, 3, 3] arrays."""
    a = np.pad(x.reshape(box + (1,)), ((1, 1), (1, 1), (1, 1), (0, 0)))
    for k, w in enumerate(ws):
        out = np.zeros(box + (w.shape[0],))
        for i in range(3):
            for j in range(3):
                for l in range(3):
                    out += a[i:i + box[0], j:j + box[1], l:l + box[2]] @ w[:, :, i, j, l].T
        if relu and k < 2:
            out = np.maximum(out, 0)
        a = np.pad(out, ((1, 1), (1, 1), (1, 1), (0, 0)))
    return out[..., 0].reshape(-1)


@pytest.mark.parametrize("box,nb,pad", [((1, 1, 1), 1, 0), ((3, 5, 7), 2, 1), ((6, 4, 9), 15, 0), ((5, 3, 8), 16, 2),
                                        ((4, 6, 5), 17, 0), ((2, 7, 5), 5, 1), ((3, 8, 4), 8, 0), ((7, 3, 6), 33, 1), ((3, 4, 10), 64, 0)])
def test_net_edges(box, nb, pad):
    from paper_1306_2953_gb300 import _lib, api
    import ctypes
    g = api.Grid.box(*box, 0.3, order=1)           # lexicographic: points in box order
    H = api.Hamiltonian(g, np.zeros(g.npts))
    rng = np.random.default_rng(nb)
    full = torch.from_numpy(rng.uniform(-1, 1, (g.npts, nb + 2 * pad)).astype(np.float32)).cuda()
    R, W = full[:, pad:pad + nb], torch.full_like(full, 7.0)
    ws = wl.conv_init(3)
    w = torch.from_numpy(np.concatenate([a.reshape(-1) for a in ws])).cuda()
    out = W[:, pad:pad + nb]
    _lib.call("rs_precond_apply", H._h, ctypes.c_void_p(w.data_ptr()), ctypes.c_void_p(R.data_ptr()), R.stride(0),
              ctypes.c_void_p(out.data_ptr()), out.stride(0), nb, api._stream())
    got = out.double().cpu().numpy()
    wq = [torch.from_numpy(a).to(torch.bfloat16).double().numpy() for a in ws]
    r = R.cpu().numpy()
    for k in range(nb):
        rms = np.sqrt(np.mean(r[:, k].astype(np.float64) ** 2))
        x = torch.from_numpy(r[:, k] * np.float32(1.0 / rms)).to(torch.bfloat16).double().numpy()
        ref = rms * _net(box, x, wq, True)
        mag = rms * _net(box, np.abs(x), [np.abs(a) for a in wq], False)
        assert np.all(np.abs(got[:, k] - ref) <= 3 * 216 * 2.0 ** -23 * mag)
    o = W.cpu().numpy()
    assert np.all(o[:, :pad] == 7.0) and np.all(o[:, pad + nb:] == 7.0)
