"""Enumeration and read-back of materialised spaces at their edges: ranges on
both sides of the size from which they are converted on the device, odd
parameter counts, spaces with and without a constrained-index table, and raw
sizes that end inside a tile or a run."""
import numpy as np
import pytest

import workloads as W
from oracle import space as ospace

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2102_05297_gb300 import ktune
    return ktune


def make(radices, code):
    return W.SpaceDesc("edge", ["p%d" % j for j in range(len(radices))],
                       [[i + 1 for i in range(r)] for r in radices], code)


SPACES = [
    ([3], []),                                                      # three raw indices
    ([5, 7, 11, 13, 3], W.c_divides(1, 3)),                         # a table; 15,015 raw
    ([16, 16, 17 - 1, 5], W.c_product_le([0, 1, 2], 400)),          # 20,480 raw
    ([13, 11, 9, 7, 5, 3], W.c_sum_le([0, 1, 2, 3, 4, 5], 24)),     # too wide for windows: 135,135 raw
    ([16, 16, 16, 16, 3], W.c_product_le([0, 1, 2, 3], 5000)),      # 65,536 combinations; 196,608 raw
    ([9] * 5 + [2, 2], W.c_sum_le([0, 1, 2, 3, 4], 9) + W.c_divides(5, 6)),   # past the table's size; 236,196 raw
]


@pytest.mark.parametrize("radices,code", SPACES)
def test_enumeration_and_ranges(kt, radices, code):
    desc = make(radices, code)
    ref = ospace.enumerate_valid(desc)
    sp = kt.Space.from_desc(desc)
    assert sp.count() == (len(ref), desc.n_raw)
    raw, dig = sp.valid_raw(), sp.valid_digits()
    np.testing.assert_array_equal(raw, ref)
    np.testing.assert_array_equal(dig, ospace.decode(desc.radices, ref))
    n = len(ref)
    for first, count in ((0, 1), (n - 1, 1), (n // 3, min(n - n // 3, 8191)), (1, min(n - 1, 8192)),
                         (0, min(n, 8193)), (n, 0)):
        np.testing.assert_array_equal(sp.valid_raw(first, count), ref[first:first + count])
        np.testing.assert_array_equal(sp.valid_digits(first, count), dig[first:first + count])
    # on the fly the same count, and the same first configuration for a seed
    otf = kt.Space.from_desc(desc, flags=kt.KTUNE_ON_THE_FLY)
    assert otf.count() == sp.count()
