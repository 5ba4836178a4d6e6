"""Failure detection of the contraction kernels without a GPU fault: their
bounded waits are given a limit of zero tests, so that every one gives up at once.
The kernels return; no result that was not computed keeps a finite value, and the
calls that have a status word return RS_ETIMEOUT.  With the default limit the
same calls are right again.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def limit():
    from paper_1306_2953_gb300 import _lib
    yield lambda overlap=-1, rotation=-1: _lib.call("rs_contraction_wait_limit", overlap, rotation)
    _lib.call("rs_contraction_wait_limit", -1, -1)


def _block(n, cols, dtype, seed=1):
    return torch.from_numpy(np.random.default_rng(seed).uniform(-1, 1, (n, cols))).to(dtype).cuda()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(5, 5), (130, 70), (257, 20)])
def test_overlap_wait(limit, dtype, nx, ny):
    from paper_1306_2953_gb300 import api
    t = torch.float64 if dtype == "f64" else torch.float32
    g = api.Grid.box(31, 31, 32, 0.3)
    X, Y = _block(g.npts, nx, t), _block(g.npts, ny, t, 2)
    limit(overlap=0)
    assert bool(api.overlap(g, X, Y).isnan().all())
    limit()
    S, ref = api.overlap(g, X, Y), g.dV * (X.double().T @ Y.double())
    assert (S - ref).abs().max() <= 1e-12 * g.npts * g.dV


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [20, 66, 300, 600])
def test_digit_rotation_wait(limit, dtype, n):
    """Through the orthonormalisation, whose factor is right: every row tile of
    every CTA, and not the first ones alone, holds NaN."""
    from paper_1306_2953_gb300 import api
    t = torch.float64 if dtype == "f64" else torch.float32
    g = api.Grid.box(31, 31, 32, 0.3)
    P = _block(g.npts, n, t)
    limit(rotation=0)
    C = api.orthonormalize(g, P)
    assert bool(C.isfinite().all()) and bool(P.isnan().all())
    limit()
    P = _block(g.npts, n, t)
    api.orthonormalize(g, P)
    S = g.dV * (P.double().T @ P.double())
    assert (S - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max() <= (1e-11 if dtype == "f64" else 1e-4)


@pytest.mark.parametrize("n,m,in_place", [(20, 40, True), (64, 300, True), (200, 100, False), (33, 130, False)])
def test_piece_rotation_wait(limit, n, m, in_place):
    from paper_1306_2953_gb300 import _lib, api
    npts = 40_000
    buf = _block(npts, max(n, m), torch.float32)
    X, C = buf[:, :n], _block(n, m, torch.float64, 3)
    Y = buf[:, :m] if in_place else torch.zeros((npts, m), device="cuda")
    x = X.double()
    limit(rotation=0)
    with pytest.raises(_lib.RsError) as e:
        api.rotate(X, C, Y=Y)
    assert e.value.code == _lib.RS_ETIMEOUT and bool(Y.isnan().all())
    limit()
    X.copy_(x.float())
    api.rotate(X, C, Y=Y)
    assert ((Y.double() - x @ C).abs() <= 2e-6 * (x.abs() @ C.abs())).all()


@pytest.mark.parametrize("nx,ny", [(5, 5), (130, 70), (300, 300)])
def test_piece_overlap_wait(limit, nx, ny):
    from paper_1306_2953_gb300 import _lib, api
    from paper_1306_2953_gb300.api import _c, _stream
    g = api.Grid.box(31, 31, 32, 0.3)
    X, Y = _block(g.npts, nx, torch.float32), _block(g.npts, ny, torch.float32, 2)
    S = torch.zeros((nx, ny), dtype=torch.float64, device="cuda")
    work = api.tc_workspace(nx, ny, g.npts)
    args = (g._h, _c(X.data_ptr()), nx, nx, _c(Y.data_ptr()), ny, ny, _c(S.data_ptr()), ny, _c(work.data_ptr()), _stream(None))
    limit(overlap=0)
    with pytest.raises(_lib.RsError) as e:
        _lib.call("rs_overlap_block_tc", *args)
    assert e.value.code == _lib.RS_ETIMEOUT and bool(S.isnan().all())
    limit()
    _lib.call("rs_overlap_block_tc", *args)
    assert ((S - g.dV * (X.double().T @ Y.double())).abs() <= 2e-6 * g.dV * (X.double().abs().T @ Y.double().abs())).all()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("which", ["overlap", "rotation"])
def test_solver_wait(limit, dtype, which):
    from paper_1306_2953_gb300 import _lib, api
    t = torch.float64 if dtype == "f64" else torch.float32
    g = api.Grid.box(20, 19, 18, 0.4)
    H = api.Hamiltonian(g, np.linspace(-1, 1, g.npts))
    S = api.Solver(H, _block(g.npts, 32, t), 16, 1e-6)
    S.step()
    limit(**{which: 0})
    with pytest.raises(_lib.RsError) as e:
        S.step()
    assert e.value.code == _lib.RS_ETIMEOUT
