"""32-bit instances of a mixed-path batch do not depend on the element type of their neighbours."""
import numpy as np
import pytest

from paper_2601_19650_gb300 import _cbc

from test_parity_gpu import _apply_batched
from test_steady_gpu import _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("narrow,wide", [(np.float32, np.float64), (np.complex64, np.complex128)])
def test_neighbours_of_other_types(narrow, wide):
    over = dict(L=8, chi=8, D=3, max_bond=6)
    small = [_problem(narrow, None, seed=j, **over) for j in range(3)]
    big = [_problem(narrow, wide, seed=10 + j, **over) for j in range(2)]
    alone, _ = _apply_batched(small, _cbc.CBC_PREC_MIXED)
    among, _ = _apply_batched([big[0], small[0], small[1], big[1], small[2]], _cbc.CBC_PREC_MIXED)
    for a, b in zip(alone, [among[1], among[2], among[4]]):
        assert list(a[1]) == list(b[1])
        for x, y in zip(a[0], b[0]):
            assert np.array_equal(x, y)
