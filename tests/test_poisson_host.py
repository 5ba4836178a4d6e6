"""Argument errors of the Hartree solver, which need no GPU."""
import pytest

from paper_1306_2953_gb300 import _lib, api


@pytest.mark.parametrize("box,n", [((700, 1, 1), 1458), ((1, 800, 2), 864), ((1, 1, 500), 1024)])
def test_too_long_an_axis_is_named(box, n):
    """The cube's axis has the smallest 2^p 3^q >= (e - 1) + ceil(sqrt(D2) + 1) + 1 points
    (e: the box's extent, D2: its diagonal's square); more than 768 are refused, at the first such axis."""
    with pytest.raises(_lib.RsError) as e:
        api.Poisson(api.Grid.box(*box, 0.3))
    assert e.value.code == _lib.RS_EINVAL
    assert f"cube of {n} points along an axis exceeds 768" in str(e.value)
