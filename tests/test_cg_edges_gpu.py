"""Workspace and operand placement of the shifted-Poisson conjugate gradients."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _call(H, B, X, n_iter, shift):
    """The C entry with a workspace that starts `shift` bytes into a 256-byte line."""
    from paper_1306_2953_gb300 import _lib, api
    n, code = B.shape[1], api.dtype_code(B)
    work = torch.empty(int(_lib.lib().rs_cg_workspace_bytes(B.shape[0], n, code)) + 16, dtype=torch.uint8, device="cuda")
    _lib.call("rs_shifted_poisson_cg", H._h, ctypes.c_void_p(B.data_ptr()), ctypes.c_void_p(X.data_ptr()), B.stride(0), n,
              n_iter, code, ctypes.c_void_p(work.data_ptr() + shift), api._stream())


@pytest.mark.parametrize("dtype,n,shift", [("f32", 16, 4), ("f32", 16, 8), ("f32", 2, 4), ("f64", 4, 8), ("f64", 2, 8)])
def test_misaligned_workspace_is_refused(dtype, n, shift):
    """The H psi kernels read rows 16 bytes (or a row) at a time, so a workspace
    off such a boundary is refused; without iterations it is not used and X = 0."""
    from paper_1306_2953_gb300 import _lib, api
    g = api.Grid.box(9, 8, 7, 0.3)
    H = api.Hamiltonian(g, np.ones(g.npts))
    B = torch.ones((g.npts, n), dtype=torch.float64 if dtype == "f64" else torch.float32, device="cuda")
    X = torch.full_like(B, 3.0)
    with pytest.raises(_lib.RsError) as e:
        _call(H, B, X, 3, shift)
    assert e.value.code == _lib.RS_EINVAL
    _call(H, B, X, 0, shift)
    assert not X.any()


def test_workspace_aligned_to_one_row_is_taken():
    """One FP32 column needs four bytes, wherever it starts."""
    from paper_1306_2953_gb300 import api
    g = api.Grid.box(9, 8, 7, 0.3)
    H = api.Hamiltonian(g, np.ones(g.npts))
    B = torch.from_numpy(np.random.default_rng(1).standard_normal((g.npts, 1)).astype(np.float32)).cuda()
    X, Y = torch.empty_like(B), torch.empty_like(B)
    _call(H, B, X, 6, 0)
    _call(H, B, Y, 6, 4)
    assert (X - Y).abs().max() <= 1e-6 * X.abs().max() and X.abs().max() > 0
