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


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("scales", [(1, 1e-5, 1, 1e-8), (1e-6, 1, 1e3, 1e-12), (1e20, 1e-15, 1e-3, 1)])
@pytest.mark.parametrize("n", [4, 40, 66, 300])
def test_rotation_of_columns_of_different_size(dtype, scales, n):
    """Orthonormalisation of columns whose sizes differ: Psi <- Psi U^-1 multiplies
    each by about the inverse of its size, so every one counts in full.
    Tolerance: the digits resolve s bits below the largest entry of a row of the
    columns brought to one size by powers of two, r_k, and of a column of U^-1 with its
    rows taken the other way; each of the n products is off by at most 8 * 2^-s of
    these.  The reference's sums are within n * 2^-53 of the sum of products, the
    result is rounded once."""
    from paper_1306_2953_gb300 import api
    t, s, u = (torch.float64, 62, 2.0 ** -53) if dtype == "f64" else (torch.float32, 38, 2.0 ** -24)
    g = api.Grid.box(31, 31, 32, 0.3)
    rng = np.random.default_rng(n)
    size = np.array([scales[k % 4] for k in range(n)])
    P = torch.from_numpy(rng.uniform(-1, 1, (g.npts, n)) * size).to(t).cuda()
    x = P.double().clone()
    C = api.orthonormalize(g, P)
    ref = x @ C
    r = torch.exp2(torch.floor(torch.log2(x.abs().amax(0))))
    tol = ((n + 8) * 2.0 ** -53 * (x.abs() @ C.abs()) + 2 * u * ref.abs() +
           8 * n * 2.0 ** -s * (x.abs() / r).amax(1)[:, None] * (r[:, None] * C.abs()).amax(0)[None, :])
    assert bool(((P.double() - ref).abs() <= tol).all())


@pytest.mark.parametrize("dtype,scales", [("f64", (1e150, 1.0, 1e-150, 1e5)), ("f32", (1e30, 1.0, 1e-25, 1e5))])
@pytest.mark.parametrize("n", [40, 66])
def test_rotation_of_columns_too_far_apart_for_the_digits(dtype, scales, n):
    """Sizes further apart than the digits' scaling reaches: plain sums.
    Tolerance: n terms in FP64 here and in the reference, one rounding to the type."""
    from paper_1306_2953_gb300 import api
    t, u = (torch.float64, 2.0 ** -53) if dtype == "f64" else (torch.float32, 2.0 ** -24)
    g = api.Grid.box(13, 12, 11, 0.3)
    size = np.array([scales[k % 4] for k in range(n)])
    P = torch.from_numpy(np.random.default_rng(n).uniform(-1, 1, (g.npts, n)) * size).to(t).cuda()
    x = P.double().clone()
    C = api.orthonormalize(g, P)
    ref, mag = x @ C, x.abs() @ C.abs()
    assert bool(((P.double() - ref).abs() <= (2 * (n + 8) * 2.0 ** -53 + 2 * u) * mag).all())


def test_rotation_of_zero_rows():
    """Rows of zeros (whole tiles and parts) stay zero, beside columns of two sizes."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(31, 31, 32, 0.3)
    x = np.random.default_rng(3).uniform(-1, 1, (g.npts, 70)) * np.array([1e-7 if k % 3 else 1.0 for k in range(70)])
    x[1000:5000] = 0
    P = torch.from_numpy(x).cuda()
    C = api.orthonormalize(g, P)
    assert not P[1000:5000].any()
    ref = torch.from_numpy(x).cuda() @ C
    assert (P - ref).abs().max() <= 1e-13 * ref.abs().max()
