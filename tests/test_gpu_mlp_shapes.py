"""The MLP forward at the edges of its tiles: ragged row counts around the
256-row tiles and their halves, feature layers of one to several weight chunks,
counter counts around the output layer's padding, and scores of every
configuration from those predictions."""
import numpy as np
import pytest

import workloads as W
from oracle import expert as oexpert, mlp as omlp, score as oscore

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2102_05297_gb300 import ktune
    return ktune


def space(radices):
    return W.SpaceDesc("edge", ["p%d" % j for j in range(len(radices))],
                       [[1 << i if r <= 8 else i + 1 for i in range(r)] for r in radices], [])


def setup(kt, radices, K, seed):
    desc = space(radices)
    roles = (W.LAYOUT_40 + [W.ROLE["INERT"]] * 24)[:K] if K != 16 else W.layout(16)
    sp = kt.Space.from_desc(desc)
    ranges = np.linspace(1.0, 50.0, K).astype(np.float32)
    m = kt.Mlp(sp, roles, ranges, max_batch=16)
    p = omlp.init_params(m.F, K, seed=seed)
    rng = np.random.default_rng(seed)
    for k in ("b1", "b2", "b3", "b4"):
        p[k] = (rng.standard_normal(p[k].shape) * 0.1).astype(np.float32)
    m.set_params(p)
    return desc, roles, sp, ranges, m, p


# F: 16 and 48 (one short chunk), 80 and 96 (a chunk and a tail)
@pytest.mark.parametrize("radices,K", [([2, 9], 1), ([4, 4, 3, 5, 5, 4, 2], 16), ([16, 16, 16, 16], 33),
                                       ([16] * 5 + [4], 64),
                                       ([1, 2, 7, 1, 16, 11], 40)])
def test_rows_and_counters(kt, radices, K):
    desc, roles, sp, ranges, m, p = setup(kt, radices, K, 3)
    N = min(700, sp.count()[0])
    raw = np.sort(np.random.default_rng(1).choice(sp.count()[0], size=N, replace=False)).astype(np.int64)
    dig = np.stack(np.unravel_index(raw, radices), axis=1)
    whole = m.predict(raw)
    ref = omlp.predict(p, desc.values, dig, ranges)
    # one-ulp bfloat16 flips of activations, as in the prediction test of the tiny space
    scale = np.max(np.abs(ref), axis=0) + 1e-6
    assert np.all(np.max(np.abs(whole - ref), axis=0) / scale <= 5e-3)
    for n in (1, 31, 127, 128, 129, 255, 256, 257, 384, 385, 511, 513):
        if n <= N:      # a row's counters do not depend on the rows beside it
            np.testing.assert_array_equal(m.predict(raw[:n]), whole[:n])


@pytest.mark.parametrize("radices,K", [([2, 9], 25), ([4, 4, 3, 5, 5, 4, 2], 33), ([16, 16, 16, 16], 64)])
def test_scores_follow_the_predictions(kt, radices, K):
    import torch
    desc, roles, sp, ranges, m, p = setup(kt, radices, K, 5)
    n = sp.count()[0]
    s = kt.Search(sp, kt.Model.from_mlp(m), k=2, seed=1)
    counters = np.abs(np.random.default_rng(2).standard_normal(K)).astype(np.float32) * 40
    at = s.current()
    s.step(counters)
    got = torch.empty(n, dtype=torch.float32, device="cuda")
    s.scores_device(0, n, got.data_ptr())
    torch.cuda.synchronize()
    pred = m.predict(np.arange(n, dtype=np.int64))      # no constraints: ordinal = raw index
    delta = oexpert.delta_vector(roles, counters, 0.7, 1000.0).astype(np.float32)
    np.testing.assert_array_equal(got.cpu().numpy(), oscore.score_fp32(pred[at], pred, delta))
