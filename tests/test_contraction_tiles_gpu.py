"""In-place rotations whose row tiles (128 rows) outnumber the clusters that are
resident at once, so that a cluster takes several of them: rows of the next
tile are read, and their exponents found, while this one's are written.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts", [40_000, 20_011])
@pytest.mark.parametrize("n,m", [(20, 130), (32, 256), (20, 1000), (33, 256), (256, 256)])
def test_piece_rotation_in_place_many_tiles(npts, n, m):
    """rs_rotate_block with Y = X, one stage (n <= 32) and more, column blocks in
    a cluster of two to eight CTAs.  Tolerance: as for the edges of the same
    kernel, six of nine piece products (the rest below 3 * 2^-24), C rounded to
    FP32, and at most n / 16 + 6 FP32 accumulations."""
    from paper_1306_2953_gb300 import _lib, api
    rng = np.random.default_rng(n + m)
    buf = torch.from_numpy(rng.uniform(-1, 1, (npts, m)).astype(np.float32)).cuda()
    x = buf[:, :n].double()
    C = torch.from_numpy(rng.standard_normal((n, m))).cuda()
    ref, mag = x @ C, x.abs() @ C.abs()
    work = api.tc_workspace(npts, m, n)
    _lib.call("rs_rotate_block", ctypes.c_void_p(buf.data_ptr()), m, n, ctypes.c_void_p(C.data_ptr()), m, m,
              ctypes.c_void_p(buf.data_ptr()), m, npts, ctypes.c_void_p(work.data_ptr()), api._stream())
    assert bool(((buf.double() - ref).abs() <= (2 * (n / 16 + 6) + 4) * 2.0 ** -24 * mag).all())


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [66, 300, 600])
def test_digit_rotation_in_place_many_tiles(dtype, n):
    """Psi <- Psi U^-1 for the U^-1 that the orthonormalisation returns, 30 752
    rows; 600 columns take two column blocks to a CTA.  Tolerance: the digits
    resolve s bits below the largest entry of a row of Psi and of a column of
    U^-1 (columns of one size), each product is off by at most 8 * 2^-s of
    these, the reference's own sums by n * 2^-53 of the sum of products."""
    from paper_1306_2953_gb300 import api
    t, s, u = (torch.float64, 62, 2.0 ** -53) if dtype == "f64" else (torch.float32, 38, 2.0 ** -24)
    g = api.Grid.box(31, 31, 32, 0.3)
    rng = np.random.default_rng(n)
    P = torch.from_numpy(rng.uniform(-1, 1, (g.npts, n))).to(t).cuda()
    x = P.double().clone()
    C = api.orthonormalize(g, P)
    ref = x @ C
    tol = ((n + 8) * 2.0 ** -53 * (x.abs() @ C.abs()) +
           8 * n * 2.0 ** -s * x.abs().amax(1)[:, None] * C.abs().amax(0)[None, :] + 2 * u * ref.abs())
    assert bool(((P.double() - ref).abs() <= tol).all())


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [40, 130, 300])
def test_rows_beyond_the_digits_in_many_tiles(dtype, n):
    """Rows that the digits cannot hold in some of the row tiles (one that follows
    another, the first and the last among them): those tiles take plain sums, in
    one CTA (n = 40) and in clusters.  Tolerance: a plain sum of n products in
    FP64, rounded once to the type."""
    from paper_1306_2953_gb300 import api
    t, tiny, u = (torch.float64, 1e-200, 2.0 ** -53) if dtype == "f64" else (torch.float32, 1e-30, 2.0 ** -24)
    g = api.Grid.box(31, 31, 32, 0.3)
    rng = np.random.default_rng(n)
    P = torch.from_numpy(rng.uniform(-1, 1, (g.npts, n))).to(t).cuda()
    tiles = [0, 1, 7, 100, 101, 155, 200, (g.npts - 1) // 128]
    for k in tiles:
        P[min(128 * k + 17, g.npts - 1)] *= tiny
    x = P.double().clone()
    C = api.orthonormalize(g, P)
    ref, mag = x @ C, x.abs() @ C.abs()
    err = (P.double() - ref).abs()
    for k in tiles:
        r = slice(128 * k, min(128 * k + 128, g.npts))
        assert bool((err[r] <= (2 * (n + 8) * 2.0 ** -53 + 2 * u) * mag[r]).all())
    assert bool((err <= 64 * n * u * x.abs().amax(1)[:, None] * C.abs().amax(0)[None, :]).all())
