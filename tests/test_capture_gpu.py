"""Asynchronous entry points recorded into a CUDA graph, as the first calls of a
process, and replayed on other inputs."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = """
import numpy as np, torch
from paper_1306_2953_gb300 import api
g = api.Grid.box(17, 16, 15, 0.3)
H = api.Hamiltonian(g, np.linspace(-1, 1, g.npts))
Q = api.Poisson(g)
rng = np.random.default_rng(1)
def block(n, t): return torch.from_numpy(rng.uniform(-1, 1, (g.npts, n))).to(t).cuda()
for t in (torch.float64, torch.float32):
    X, Y = block(33, t), block(70, t)
    P, HP = block(32, t), torch.empty((g.npts, 32), dtype=t, device="cuda")
    n, vh = block(1, torch.float64)[:, 0].contiguous(), torch.empty(g.npts, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    G = torch.cuda.CUDAGraph()
    with torch.cuda.graph(G):
        S = api.overlap(g, X, Y)
        H.apply(P, HP)
        Q.solve(n, vh)
    for k in range(2):
        X.copy_(block(33, t)); P.copy_(block(32, t)); n.copy_(block(1, torch.float64)[:, 0])
        G.replay()
        torch.cuda.synchronize()
        s, hp, v = S.clone(), HP.clone(), vh.clone()
        tol = 1e-12 if t == torch.float64 else 1e-5
        assert (s - g.dV * (X.double().T @ Y.double())).abs().max() <= 1e-12 * g.npts * g.dV, "overlap"
        assert (hp - H.apply(P)).abs().max() <= tol * hp.abs().max(), "hpsi"
        assert (v - Q.solve(n)).abs().max() <= 1e-12 * v.abs().max(), "poisson"
print("captured ok")
"""


def test_first_calls_in_a_capture():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, env=dict(os.environ, PYTHONPATH=root),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured ok" in r.stdout, r.stdout + r.stderr
