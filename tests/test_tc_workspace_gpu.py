"""Workspace checks of the tensor-core contractions of FP32 orbitals."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [1, 4, 8])
def test_misaligned_workspace_is_refused(shift):
    from paper_1306_2953_gb300 import _lib, api
    g = api.Grid.box(5, 4, 3, 0.3)
    X = torch.ones((g.npts, 8), device="cuda")
    C = torch.ones((8, 8), dtype=torch.float64, device="cuda")
    S = torch.empty((8, 8), dtype=torch.float64, device="cuda")
    p = lambda t, o=0: ctypes.c_void_p(t.data_ptr() + o)
    for call in (lambda w: _lib.call("rs_rotate_block", p(X), 8, 8, p(C), 8, 8, p(Y), 8, g.npts, p(w, shift), api._stream()),
                 lambda w: _lib.call("rs_overlap_block_tc", g._h, p(X), 8, 8, p(X), 8, 8, p(S), 8, p(w, shift), api._stream())):
        Y = torch.full_like(X, 5.0)
        work = torch.empty(api.tc_workspace(g.npts, 64, 64).numel() + 64, dtype=torch.uint8, device="cuda")
        with pytest.raises(_lib.RsError) as e:
            call(work)
        assert e.value.code == _lib.RS_EINVAL
        assert bool((Y == 5.0).all())
