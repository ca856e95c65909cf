"""Read-back and creation of materialised spaces on a GPU with little memory left:
what fits beside the space itself is enough."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def kt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2102_05297_gb300 import ktune
    return ktune


class Filled:
    """All but about `left` bytes of the device's memory, held."""

    def __init__(self, left):
        self.left = left

    def __enter__(self):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.blocks = []
        while True:
            n = (torch.cuda.mem_get_info()[0] - self.left) // (2 * MB) * (2 * MB)
            if n <= 0:
                return self
            self.blocks.append(torch.empty(n, dtype=torch.uint8, device="cuda"))

    def __exit__(self, *exc):
        import torch
        self.blocks.clear()
        torch.cuda.empty_cache()


def make(kt, radices, code, flags=0):
    return kt.Space.from_desc(W.SpaceDesc("m", ["p%d" % j for j in range(len(radices))],
                                          [list(range(1, r + 1)) for r in radices], code), flags=flags)


# 5,242,880 configurations: two conversions of at most 4,194,304; with 6 MB left
# there is no room for one, with 40 MB for one of 33.6 MB but not for 41.9
@pytest.mark.parametrize("left", [6 * MB, 40 * MB])
def test_read_back_beside_a_full_device(kt, left):
    radices = [16, 16, 16, 16, 16, 5]
    sp = make(kt, radices, [])
    n = sp.count()[0]
    assert n == int(np.prod(radices))
    raw, dig = sp.valid_raw(), sp.valid_digits()
    np.testing.assert_array_equal(raw, np.arange(n))
    with Filled(left):
        np.testing.assert_array_equal(sp.valid_raw(), raw)
        np.testing.assert_array_equal(sp.valid_digits(), dig)
        np.testing.assert_array_equal(sp.valid_raw(7, n - 8), raw[7:n - 1])
    np.testing.assert_array_equal(dig, np.stack(np.unravel_index(raw, radices), axis=1))


def test_failed_allocation_is_reported_once(kt):
    """A creation that does not fit fails with KTUNE_ENOMEM, and only that one."""
    with Filled(6 * MB):
        with pytest.raises(kt.KtuneError, match="cudaMalloc"):
            make(kt, [16, 16, 16, 16, 16, 5], [])
        assert make(kt, [3, 5], []).count() == (15, 15)
    assert make(kt, [3, 5], []).count() == (15, 15)


# 2^30 raw indices, whose valid bits would take 134 MB: no room for them at all
# (81,920 configurations), or for them but not for 8.1M configurations beside them
@pytest.mark.parametrize("total,left", [(5, 48 * MB), (12, 160 * MB)])
def test_creation_without_room_for_the_valid_bits(kt, total, left):
    radices, code = [16] * 7 + [4], W.c_sum_le([0, 1, 2, 3], total)
    ref = make(kt, radices, code)
    raw = ref.valid_raw()
    ref.close()
    with Filled(left):
        sp = make(kt, radices, code)
        assert sp.count() == (len(raw), 1 << 30)
        got = sp.valid_raw()
    np.testing.assert_array_equal(got, raw)
    digits = np.stack(np.unravel_index(raw[::997], radices), axis=1)
    assert np.all(digits[:, :4].sum(axis=1) + 4 <= total)
