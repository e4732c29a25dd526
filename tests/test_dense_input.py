"""The nonzero entries that a dense check matrix is handed to the library by: numpy's own, in row-major
order, for every memory layout and size."""
import numpy as np
import pytest

from paper_2406_18655_gb300.lsd import _ones


@pytest.mark.parametrize("shape", [(0, 3), (3, 0), (1, 1), (1, 70), (70, 1), (37, 61), (300, 700)])
@pytest.mark.parametrize("layout", ["C", "F", "strided", "reversed"])
def test_entries(shape, layout):
    rng = np.random.default_rng(3)
    m, n = shape
    wide = (rng.random((2 * m, 3 * n)) < 0.2).astype(np.uint8) * 7
    h = {"C": np.ascontiguousarray(wide[:m, :n]), "F": np.asfortranarray(wide[:m, :n]),
         "strided": wide[::2, ::3], "reversed": wide[:m, :n][::-1, ::-1]}[layout]
    got, want = _ones(h), np.nonzero(h)
    for a, b in zip(got, want):
        assert a.dtype == np.int32 and a.flags.c_contiguous and np.array_equal(a, b)


def test_only_matrices():
    with pytest.raises(ValueError):
        _ones(np.zeros(4, np.uint8))
