"""Activations of the learned preconditioner beyond the FP32 range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [(17, 18, 19), (27, 28, 29)])
@pytest.mark.parametrize("nb", [4, 12, 16, 32])
def test_infinite_activations_stay_infinite(nb, d):
    """One spike per column overflows the first layer's first channel: the output
    is infinite within the network's reach of three points and finite elsewhere, as the network
    in FP64 with every layer's output cast to FP32 says.  Tolerance of the finite values: FP32 sums of
    8 * 27 products and BF16 rounding of the input (2^-9, of either neighbour)."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(*d, 0.3)
    H = api.Hamiltonian(g, np.zeros(g.npts))
    rng = np.random.default_rng(nb)
    ijk = g.ijk()
    u = ijk - ijk.min(0)
    w1, w2, w3 = np.full((8, 1, 27), 0.125), np.full((8, 8, 27), 2.0 ** -7), np.full((1, 8, 27), 2.0 ** -7)
    w1[0] = 2.0 ** 123
    w = torch.from_numpy(np.concatenate([w1.ravel(), w2.ravel(), w3.ravel()]).astype(np.float32)).cuda()
    box = 1e-3 * rng.uniform(0.5, 1, (nb, *d))
    at = [(3 + k % 9, 5 + k % 7, 4 + k % 11) for k in range(nb)]
    for k, p in enumerate(at):
        box[(k, *p)] = 1.0
    R = box.astype(np.float32)[:, u[:, 0], u[:, 1], u[:, 2]].T.copy()
    W = api.precond_apply(H, w, torch.from_numpy(R).cuda()).double().cpu().numpy()

    rms = np.sqrt((R.astype(np.float64) ** 2).mean(0))
    a = torch.from_numpy(box.astype(np.float32) / rms[:, None, None, None].astype(np.float32))
    a = a.to(torch.bfloat16).double()[:, None]
    with np.errstate(all="ignore"):
        for wl, relu in ((w1, True), (w2, True), (w3, False)):
            k = torch.from_numpy(wl.reshape(wl.shape[0], wl.shape[1], 3, 3, 3))
            big = torch.isinf(a)
            fin = torch.nn.functional.conv3d(torch.where(big, 0.0, a), k, padding=1)
            hit = torch.nn.functional.conv3d(big.double(), torch.ones_like(k), padding=1) > 0   # (all weights are positive)
            a = torch.where(hit, float("inf"), fin).float().double()
            a = torch.relu(a) if relu else a
    ref = a[:, 0].numpy()[:, u[:, 0], u[:, 1], u[:, 2]].T * rms
    assert np.isinf(ref).any() and np.isfinite(ref).any()
    assert np.array_equal(np.isinf(W), np.isinf(ref))
    f = np.isfinite(ref)
    assert np.all(np.abs(W - ref)[f] <= 2.0 ** -8 * np.abs(ref)[f])
