"""Overlaps and rotations by integer digits on the tensor cores (digits.cu) at
the edges of their tiles (128 x 32 / 64 results, 32 points per stage, 256 per
readout), for unaligned and strided operands, and for columns and rows that
the digits cannot hold.

Tolerances.  The operands are rounded to s bits below the largest entry of
their column (overlap; row of X and column of C in the rotation): s = 62
(FP64), 54 (FP32 overlap), 38 (FP32 rotation), and the digit products left out
are below the same size; each of the K products is therefore off by at most
8 * 2^-s of the product of those largest entries.  The result is rounded
once to its type, and numpy's own sum of K products is within
K * 2^-53 * sum |x y|.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _block(n, cols, seed, dtype, pad):
    """A column slice of a wider device array, starting `pad` columns in."""
    rng = np.random.default_rng(seed)
    full = rng.uniform(-1, 1, (n, cols + 2 * pad)) * np.exp(rng.uniform(-6, 0, (n, 1)))
    t = torch.from_numpy(full).to(dtype).cuda()
    return t[:, pad:pad + cols]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("box", [(5, 3, 2), (8, 8, 4), (9, 7, 13)])
@pytest.mark.parametrize("nx,ny,pad", [(1, 1, 0), (127, 31, 1), (128, 32, 0), (129, 33, 3), (40, 65, 2), (257, 130, 0)])
def test_overlap_edges(dtype, box, nx, ny, pad):
    from paper_1306_2953_gb300 import api
    t, s = (torch.float64, 62) if dtype == "f64" else (torch.float32, 54)
    g = api.Grid.box(*box, 0.3)
    K = g.npts
    X, Y = _block(K, nx, 1, t, pad), _block(K, ny, 2, t, pad)
    for A, B in ((X, Y), (X, X)):
        S = api.overlap(g, A, B).cpu().numpy()
        a, b = A.double().cpu().numpy(), B.double().cpu().numpy()
        ref = g.dV * (a.T @ b)
        tol = g.dV * ((K + 8) * 2.0 ** -53 * (np.abs(a).T @ np.abs(b)) +
                      8 * K * 2.0 ** -s * np.abs(a).max(0)[:, None] * np.abs(b).max(0)[None, :])
        assert np.all(np.abs(S - ref) <= tol)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,pad", [(2, 0), (31, 1), (32, 0), (33, 0), (64, 2), (65, 3), (129, 0), (513, 0)])
def test_rotation_edges(dtype, n, pad):
    """In place, through the orthonormalisation: Psi <- Psi U^-1 for the U^-1 it returns."""
    from paper_1306_2953_gb300 import api
    t, s, u = (torch.float64, 62, 2.0 ** -53) if dtype == "f64" else (torch.float32, 38, 2.0 ** -24)
    g = api.Grid.box(11, 9, 10, 0.3)
    P = _block(g.npts, n, 3, t, pad)
    x = P.double().cpu().numpy()
    C = api.orthonormalize(g, P).cpu().numpy()
    ref = x @ C
    tol = ((n + 8) * 2.0 ** -53 * (np.abs(x) @ np.abs(C)) +
           8 * n * 2.0 ** -s * np.abs(x).max(1)[:, None] * np.abs(C).max(0)[None, :] + 2 * u * np.abs(ref))
    assert np.all(np.abs(P.double().cpu().numpy() - ref) <= tol)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_values_beyond_the_digits(dtype):
    """Infinities and NaN spread as in a plain sum, very small columns keep
    their accuracy, zero columns give zeros."""
    from paper_1306_2953_gb300 import api
    t, tiny = (torch.float64, 1e-200) if dtype == "f64" else (torch.float32, 1e-30)
    g = api.Grid.box(9, 8, 7, 0.3)
    X, Y = _block(g.npts, 70, 5, t, 0), _block(g.npts, 150, 6, t, 0)
    X[3, 5], X[4, 66], Y[7, 9], Y[8, 140] = float("inf"), float("nan"), float("-inf"), float("nan")
    X[:, 8] *= tiny
    Y[:, 20] = 0
    S = api.overlap(g, X, Y).cpu().numpy()
    a, b = X.double().cpu().numpy(), Y.double().cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = g.dV * np.array([[np.sum(a[:, i] * b[:, j]) for j in range(150)] for i in range(70)])
    fin = np.isfinite(ref)
    assert np.array_equal(np.isnan(S), np.isnan(ref)) and np.array_equal(S[np.isinf(ref)], ref[np.isinf(ref)])
    assert np.all(S[:5, 20] == 0)
    assert np.abs(S[8] - ref[8])[fin[8]].max() <= 1e-12 * np.abs(ref[8][fin[8]]).max()
    # a row beyond the range in the rotation (its tile takes the plain sums)
    P = _block(g.npts, 40, 7, t, 0)
    P[200] *= tiny
    x = P.double().cpu().numpy()
    C = api.orthonormalize(g, P).cpu().numpy()
    ref = x @ C
    err = np.abs(P.double().cpu().numpy() - ref)
    u = 2.0 ** -52 if dtype == "f64" else 2.0 ** -23
    assert np.all(err <= 64 * u * (np.abs(x) @ np.abs(C)))


@pytest.mark.parametrize("npts,n,m,where", [(1, 1, 1, "out"), (127, 31, 64, "out"), (129, 33, 65, "out"), (300, 40, 40, "in"),
                                            (260, 64, 130, "in"), (515, 256, 256, "in"), (200, 130, 300, "wide"),
                                            (200, 64, 64, "beside"), (300, 96, 96, "shifted"), (140, 20, 1100, "in")])
def test_piece_rotation_edges(npts, n, m, where):
    """rs_rotate_block out of place, in place (m up to and above the cluster's
    1024 columns), beside X in one array, and partly over X.  Tolerance: six of
    nine piece products (the rest below 3 * 2^-24), C rounded to FP32, and at
    most n / 16 + 6 FP32 accumulations."""
    import ctypes
    from paper_1306_2953_gb300 import _lib, api
    rng = np.random.default_rng(n + m)
    ld = {"out": n + 3, "in": max(n, m) + 1, "wide": max(n, m), "beside": n + m, "shifted": n + m}[where]
    buf = torch.from_numpy(rng.uniform(-1, 1, (npts, ld)).astype(np.float32)).cuda()
    x = buf[:, :n].double().cpu().numpy()
    C = torch.from_numpy(rng.standard_normal((n, m))).cuda()
    if where == "out":
        Y = torch.full((npts, m + 1), 7.0, device="cuda")[:, :m]
    elif where in ("in", "wide"):
        Y = buf[:, :m]
    elif where == "beside":
        Y = buf[:, n:]
    else:
        Y = buf[:, 5:5 + m]
    work = api.tc_workspace(npts, m, n)
    _lib.call("rs_rotate_block", ctypes.c_void_p(buf.data_ptr()), buf.stride(0), n, ctypes.c_void_p(C.data_ptr()), m, m,
              ctypes.c_void_p(Y.data_ptr()), Y.stride(0), npts, ctypes.c_void_p(work.data_ptr()), api._stream())
    c = C.cpu().numpy()
    ref, mag = x @ c, np.abs(x) @ np.abs(c)
    u = 2.0 ** -24
    assert np.all(np.abs(Y.double().cpu().numpy() - ref) <= (2 * (n / 16 + 6) + 4) * u * mag)


@pytest.mark.parametrize("box", [(5, 3, 2), (8, 8, 4), (41, 40, 17)])
@pytest.mark.parametrize("nx,ny,pad", [(1, 1, 0), (127, 31, 1), (128, 64, 0), (129, 65, 3), (257, 130, 0)])
def test_piece_overlap_edges(box, nx, ny, pad):
    """rs_overlap_block_tc.  Tolerance: six of nine piece products (the rest
    below 3 * 2^-24), one FP32 accumulation (2^-23 where truncated) per product
    and 16 of at most 2048 points."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(*box, 0.3)
    X, Y = _block(g.npts, nx, 4, torch.float32, pad), _block(g.npts, ny, 5, torch.float32, pad)
    for A, B in ((X, Y), (X, X)):
        S = api.overlap_tc(g, A, B).cpu().numpy()
        a, b = A.double().cpu().numpy(), B.double().cpu().numpy()
        steps = 6 * (min(g.npts, 2048) // 16 + 4)
        assert np.all(np.abs(S - g.dV * (a.T @ b)) <= g.dV * (2 * steps + 4) * 2.0 ** -24 * (np.abs(a).T @ np.abs(b)))


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 129, 160, 161, 257])
def test_factor_and_inverse_edges(n):
    """The triangular factor's inverse at the edges of its kernels (32, 64, 128
    and 256 columns; one CTA up to 160): C^T S C = 1 and C upper triangular.
    Tolerance: n rounded terms in each of the factor, the inverse and numpy's
    products, times the condition of S (below 2)."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(24, 24, 24, 0.3)
    rng = np.random.default_rng(n)
    P = torch.from_numpy(rng.standard_normal((g.npts, n))).cuda()
    p = P.cpu().numpy()
    S = g.dV * (p.T @ p)
    assert n == 1 or np.linalg.cond(S) < 2
    C = api.orthonormalize(g, P).cpu().numpy()
    assert np.array_equal(C, np.triu(C))
    assert np.abs(C.T @ S @ C - np.eye(n)).max() <= 16 * (n + 8) * 2.0 ** -53


@pytest.mark.parametrize("n,bad", [(5, 3), (48, 47), (130, 64), (200, 130)])
def test_dependent_column_is_refused(n, bad):
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(12, 12, 12, 0.3)
    P = torch.from_numpy(np.random.default_rng(n).standard_normal((g.npts, n))).cuda()
    P[:, bad] = 0.0
    with pytest.raises(Exception):
        api.orthonormalize(g, P)
