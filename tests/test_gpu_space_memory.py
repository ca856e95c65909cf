"""Read-back and creation of materialised spaces on a GPU with little memory left:
what fits beside the space itself is enough.

The cases fill the device from processes of their own: what a driver holds back for the
kernels that a process has run before gives way under pressure, and would be room that
they do not mean to leave.  (Memory that others have just given back may turn up later:
a case then has more room than it means to leave, never less.)"""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20


class Filled:
    """All but about `left` bytes of the device's memory, held."""

    def __init__(self, left):
        self.left = left

    def __enter__(self):
        import torch
        torch.cuda.synchronize()
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


def make(radices, code):
    import workloads as W
    from paper_2102_05297_gb300 import ktune
    return ktune.Space.from_desc(W.SpaceDesc("m", ["p%d" % j for j in range(len(radices))],
                                             [list(range(1, r + 1)) for r in radices], code))


# 5,242,880 configurations: two conversions of at most 4,194,304; with 6 MB left
# there is no room for one, with 40 MB for one of 33.6 MB but not for 41.9
def read_back(left):
    radices = [16, 16, 16, 16, 16, 5]
    sp = make(radices, [])
    n = sp.count()[0]
    assert n == int(np.prod(radices))
    raw, dig = sp.valid_raw(), sp.valid_digits()
    np.testing.assert_array_equal(raw, np.arange(n))
    with Filled(left):
        np.testing.assert_array_equal(sp.valid_raw(), raw)
        np.testing.assert_array_equal(sp.valid_digits(), dig)
        np.testing.assert_array_equal(sp.valid_raw(7, n - 8), raw[7:n - 1])
    np.testing.assert_array_equal(dig, np.stack(np.unravel_index(raw, radices), axis=1))


def reported_once():
    """A creation that does not fit (16^9 configurations, 550 GB) fails with
    KTUNE_ENOMEM, and only that one."""
    from paper_2102_05297_gb300 import ktune
    with pytest.raises(ktune.KtuneError, match="cudaMalloc"):
        make([16] * 9, [])
    assert make([3, 5], []).count() == (15, 15)


# 2^30 raw indices, whose valid bits would take 134 MB: no room for them at all
# (81,920 configurations), or for them but not for 8.1M configurations beside them
def no_room_for_bits(total, left):
    import workloads as W
    radices, code = [16] * 7 + [4], W.c_sum_le([0, 1, 2, 3], total)
    ref = make(radices, code)
    raw = ref.valid_raw()
    ref.close()
    with Filled(left):
        sp = make(radices, code)
        assert sp.count() == (len(raw), 1 << 30)
        got = sp.valid_raw()
    np.testing.assert_array_equal(got, raw)
    digits = np.stack(np.unravel_index(raw[::997], radices), axis=1)
    assert np.all(digits[:, :4].sum(axis=1) + 4 <= total)


@pytest.mark.gpu
@pytest.mark.parametrize("case", ["read_back(6 * MB)", "read_back(40 * MB)", "reported_once()",
                                  "no_room_for_bits(5, 48 * MB)", "no_room_for_bits(12, 160 * MB)"])
def test_little_memory_left(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.empty_cache()
    code = ("import sys; sys.path[:0] = [%r, %r]; import test_gpu_space_memory as t; MB = t.MB; t.%s"
            % (ROOT, os.path.dirname(os.path.abspath(__file__)), case))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
