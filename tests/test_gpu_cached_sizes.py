"""Cached tree steps where the leaf columns end inside a group of eight
configurations, where a CTA has no group or one, and where only some of the
counters' term tables fit shared memory, against steps that predict again."""
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


@pytest.mark.parametrize("radices,K,depth", [
    ((3,), 16, 4), ((7, 9, 11), 16, 8), ((16, 16, 5, 3), 40, 12), ((15, 15, 15, 15), 40, 14),
    ((13, 11, 16, 16, 15), 32, 12), ((16, 16, 16, 16, 10), 16, 13)])
def test_cached_equals_uncached(kt, radices, K, depth):
    import torch
    desc = W.SpaceDesc("c", ["p%d" % j for j in range(len(radices))],
                       [list(range(1, r + 1)) for r in radices], [])
    roles = W.layout(K)
    gpu = SyntheticGPU(desc, roles, seed=6)
    sp = kt.Space.from_desc(desc)
    n = sp.count()[0]
    m = kt.Model(sp, random_model(desc.radices, roles, depth=depth, seed=depth))
    k = min(4, n - 1)
    a, b = (kt.Search(sp, m, k=k, seed=8) for _ in range(2))
    b.set_cached(True)
    for _ in range(2):
        c = gpu.evaluate(np.stack(np.unravel_index([a.current()], radices), axis=1))[0][0]
        out = []
        for s in (a, b):
            try:
                raw, sc = s.step(c)
            except kt.KtuneError as e:
                assert n <= 2 * k + 1, e
                return
            sd = torch.zeros(n, device="cuda")
            torch.cuda.synchronize()
            s.scores_device(0, n, sd.data_ptr())
            torch.cuda.synchronize()
            if len(raw):
                s.report(np.arange(1, len(raw) + 1, dtype=np.float64))
            out.append((np.array(raw), np.array(sc), sd.cpu().numpy()))
        for x, y in zip(*out):
            np.testing.assert_array_equal(x, y)
