"""The gather kernel of H psi at the edges of its pieces (64 to 256 points per
CTA), for every block width, both types, several point orders and column
slices that start inside a row.

Tolerance: 27 + 4 k rounded terms per element (k atoms covering the point)
of the oracle's term magnitudes, and the projection's sums (see
test_ham_gpu), 64 roundings of the local and 512 of the nonlocal magnitude.
"""
import numpy as np
import pytest

import workloads as wl
from tests.helpers import SMALL_ATOMS, SMALL_E, SMALL_H, SMALL_RADIUS, lib_to_oracle_index, oracle_system
from tests.test_ham_gpu import _term_magnitudes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nb", [1, 2, 4, 8, 16, 32, 64])
@pytest.mark.parametrize("system,order,pad", [("one", 0, 0), ("box4", -1, 4), ("box5", 1, 0), ("mol", 2, 4), ("mol", 0, 0)])
def test_gather_edges(dtype, nb, system, order, pad):
    from paper_1306_2953_gb300 import _lib, api
    if system == "mol":
        params = ("atoms", (SMALL_ATOMS, SMALL_E, SMALL_RADIUS, SMALL_H))
    else:
        params = ("box", ({"one": 1, "box4": 4, "box5": 5}[system], 0.3, 1.0))
    g_ora, H_ora, atoms, E = oracle_system(params[0], *params[1])
    if system == "mol":
        lg = api.Grid.spheres(atoms, SMALL_RADIUS, SMALL_H, order)
        proj = api.Projectors(lg, atoms, E, 1.0, 3.0)
    else:
        n = params[1][0]
        lg, proj = api.Grid.box(n, n, n, 0.3, order), None
    idx = lib_to_oracle_index(g_ora, lg.ijk())
    H = api.Hamiltonian(lg, H_ora.V[idx], proj)
    H.select_kernel(_lib.RS_KERNEL_GENERIC)
    t, u = (torch.float64, 2.0 ** -53) if dtype == "f64" else (torch.float32, 2.0 ** -24)
    ld = nb + 2 * pad
    full = torch.from_numpy(np.ascontiguousarray(wl.random_block(g_ora.npts, ld, 9)[idx])).to(t).cuda()
    out = torch.full_like(full, 7.0)
    H.apply(full[:, pad:pad + nb], out[:, pad:pad + nb], nb=nb)
    psi = np.empty((g_ora.npts, nb))
    psi[idx] = full[:, pad:pad + nb].double().cpu().numpy()
    ref = H_ora.apply(psi)[idx]
    if proj is not None:
        m_loc, m_nl = _term_magnitudes(g_ora, H_ora, psi)
        bound = u * (64.0 * m_loc[idx] + 512.0 * m_nl[idx])
    else:
        w = 9.0 * 2.85 / (2 * 0.3 ** 2)   # three axes of weights, sum of |c_j| below 3 * 2.85
        bound = np.full_like(ref, 64.0 * u * (w + np.abs(H_ora.V).max()))
    o = out.double().cpu().numpy()
    assert np.all(np.abs(o[:, pad:pad + nb] - ref) <= bound)
    assert np.all(o[:, :pad] == 7.0) and np.all(o[:, pad + nb:] == 7.0)


@pytest.mark.parametrize("box", [(1, 1, 1), (3, 2, 5), (4, 8, 16), (5, 9, 17), (23, 7, 33), (70, 12, 40)])
def test_ring_march_edges(box):
    """FP32 blocks of 32 states (the ring kernel): columns shorter than the
    star, ragged tiles, runs that are cut inside a column.  Against the FP64
    gather of the same values; tolerance 64 roundings of the terms' magnitude,
    the sum of the weights and the potential times the largest value."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(*box, 0.3)
    rng = np.random.default_rng(sum(box))
    V = rng.uniform(-2, 2, g.npts)
    H = api.Hamiltonian(g, V, None)
    psi = torch.from_numpy(rng.uniform(-1, 1, (g.npts, 64)).astype(np.float32)).cuda()
    bound = 64 * 2.0 ** -24 * (9.0 * 2.85 / (2 * 0.3 ** 2) + 2)
    for c0, nb in ((0, 32), (32, 32), (0, 64)):
        out = torch.full_like(psi, 7.0)
        H.apply(psi[:, c0:c0 + nb], out[:, c0:c0 + nb], nb=nb)
        ref = H.apply(psi[:, c0:c0 + nb].double().contiguous(), nb=nb)
        assert (out[:, c0:c0 + nb].double() - ref).abs().max().item() <= bound
    assert H.status() == 0


def test_projection_parts_repeat():
    """The projections' parts are added in a fixed order, so a block gives the
    same bits again after blocks of other widths and types on the same handle,
    one after the other without a pause, and in a replayed graph."""
    from paper_1306_2953_gb300 import _lib, api
    g_ora, H_ora, atoms, E = oracle_system("atoms", SMALL_ATOMS, SMALL_E, SMALL_RADIUS, SMALL_H)
    lg = api.Grid.spheres(atoms, SMALL_RADIUS, SMALL_H)
    H = api.Hamiltonian(lg, H_ora.V[lib_to_oracle_index(g_ora, lg.ijk())], api.Projectors(lg, atoms, E, 1.0, 3.0))
    gen = torch.Generator(device="cuda").manual_seed(3)
    blocks = [(t, nb, k) for k in (_lib.RS_KERNEL_AUTO, _lib.RS_KERNEL_GENERIC) for t in (torch.float32, torch.float64)
              for nb in (1, 4, 16, 32, 64)]
    psi = {b: torch.rand((lg.npts, b[1]), generator=gen, device="cuda", dtype=b[0]) - 0.5 for b in blocks}

    def run(out):
        for b in blocks:
            H.select_kernel(b[2])
            H.apply(psi[b], out[b], nb=b[1])

    first, again, graph = ({b: torch.empty_like(psi[b]) for b in blocks} for _ in range(3))
    run(first)
    for _ in range(3):
        run(again)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg, stream=s):
        run(graph)
    for _ in range(3):
        cg.replay()
    torch.cuda.synchronize()
    for b in blocks:
        assert torch.equal(first[b], again[b]) and torch.equal(first[b], graph[b]), b
