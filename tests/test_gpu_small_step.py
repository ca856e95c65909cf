"""Steps of small spaces as one CTA against the same search's four kernels: every
score, weight and pick, at the sizes around its configurations per thread, tree
depths from one level to one tree per staging group, and down to the last
configuration of a space."""
import numpy as np
import pytest

import workloads as W
from workloads.synth import SyntheticGPU
from workloads.trees import random_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2102_05297_gb300 import ktune
    return ktune


def both(kt, radices, K, depth, k, steps, gamma=-0.25, stream=None):
    import torch
    desc = W.SpaceDesc("s", ["p%d" % j for j in range(len(radices))],
                       [[1 << i if r <= 8 else i + 1 for i in range(r)] for r in radices], [])
    roles = W.layout(K)
    gpu = SyntheticGPU(desc, roles, seed=3)
    sp = kt.Space.from_desc(desc)
    n = sp.count()[0]
    m = kt.Model(sp, random_model(desc.radices, roles, depth=depth, seed=depth))
    a = kt.Search(sp, m, k=k, seed=5, gamma=gamma, stream=stream)
    b = kt.Search(sp, m, k=k, seed=5, gamma=gamma, stream=stream)
    b.set_fused(0)
    assert a.current() == b.current()
    left = n - 1
    for step in range(steps):
        c = gpu.evaluate(np.stack(np.unravel_index([a.current()], radices), axis=1))[0][0]
        if step == 2:
            c = c * 0          # no bottleneck: every configuration weighs the same
        (ra, sa), (rb, sb) = a.step(c), b.step(c)
        np.testing.assert_array_equal(ra, rb)
        np.testing.assert_array_equal(sa, sb)
        assert len(ra) == min(k, left)
        left -= len(ra)
        out = [torch.zeros(n, dtype=t, device="cuda") for t in (torch.float32, torch.int32) * 2]
        torch.cuda.synchronize()
        a.scores_device(0, n, out[0].data_ptr(), out[1].data_ptr(), stream)
        b.scores_device(0, n, out[2].data_ptr(), out[3].data_ptr(), stream)
        torch.cuda.synchronize()
        assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])
        x, y = a.stats(), b.stats()
        assert (x.n_scored, x.n_active, x.s_min, x.s_max) == (y.n_scored, y.n_active, y.s_min, y.s_max)
        if not len(ra):
            break
        rt = np.arange(len(ra), 0, -1, dtype=float)
        a.report(rt)
        b.report(rt)
    assert a.evaluated() == b.evaluated()
    return left


@pytest.mark.parametrize("radices", [[2], [3, 11], [7, 9, 16], [16, 8, 8], [13, 5, 16], [16, 16, 8],
                                     [13, 10, 16], [9, 5, 7, 13], [16, 16, 16], [13, 10, 16, 2]])
def test_sizes(kt, radices):
    both(kt, radices, 32, 10, 5, 4)


@pytest.mark.parametrize("depth,K", [(1, 16), (2, 40), (8, 16), (12, 40), (13, 32), (14, 32)])
def test_depths(kt, depth, K):
    import torch
    both(kt, [9, 5, 7, 3, 2], K, depth, 7, 4, stream=torch.cuda.Stream())


def test_all_of_a_space(kt):
    assert both(kt, [7, 5, 9], 16, 6, 64, 8) == 0
    both(kt, [16, 16, 8], 16, 6, 33, 6, gamma=0.5)
