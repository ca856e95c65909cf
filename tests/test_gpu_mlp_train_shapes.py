"""MLP training at the edges of its kernels' tiles: counters that leave the output
layer's columns padded and its targets unaligned, one to three chunks of feature
columns and a second tile of them, batches below a cluster's rows and beyond the slices
that the weight gradients are split into, and handles that train both.

Bounds as in test_gpu_mlp.py: two sides differ by float32 accumulation order (K 2^-22 of
sum |a b|) and by the one-ulp bfloat16 flips it causes, 2^-8 of an operand each, so 2e-2
of a tensor's largest element and 5e-3 of its norm."""
import numpy as np
import pytest

import workloads as W
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

# feature columns: 16, 96, 144 (the last over 2^32 raw indices, decoded on the fly)
RADICES = {16: [2, 9], 96: [16] * 5 + [4], 144: [16] * 8}


@pytest.fixture(scope="module")
def kt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2102_05297_gb300 import ktune
    return ktune


def setup(kt, F, K, max_batch, seed):
    radices = RADICES[F]
    desc = W.SpaceDesc("t", ["p%d" % j for j in range(len(radices))],
                       [list(range(1, r + 1)) for r in radices], [])
    sp = kt.Space.from_desc(desc, flags=kt.KTUNE_ON_THE_FLY)
    roles = (W.LAYOUT_40 + [W.ROLE["INERT"]] * 24)[:K]
    ranges = np.linspace(1.0, 50.0, K).astype(np.float32)
    m = kt.Mlp(sp, roles, ranges, max_batch=max_batch)
    assert m.F == F
    p = omlp.init_params(F, K, seed=seed)
    rng = np.random.default_rng(seed)
    for k in ("b1", "b2", "b3", "b4"):
        p[k] = (rng.standard_normal(p[k].shape) * 0.1).astype(np.float32)
    m.set_params(p)
    n = 600
    raw = rng.integers(0, desc.n_raw, size=n).astype(np.int64)
    dig = np.stack(np.unravel_index(raw, radices), axis=1)
    C = (rng.random((n, K)) * ranges).astype(np.float32)
    m.set_data(raw, C)
    return m, p, omlp.features(desc.values, dig), (C / ranges).astype(np.float32), rng


def compare(m, p, x, t, idx):
    loss, g = m.grads(idx)
    oloss, og = omlp.loss_and_grads(p, x[idx], t[idx])
    assert abs(loss - oloss) <= 1e-3 * oloss
    for k in og:
        scale = float(np.max(np.abs(og[k]))) + 1e-12
        assert float(np.max(np.abs(g[k] - og[k]))) <= 2e-2 * scale, k
        assert np.linalg.norm(g[k] - og[k]) <= 5e-3 * (np.linalg.norm(og[k]) + 1e-12), k


@pytest.mark.parametrize("F,K,B", [(16, 1, 16), (16, 64, 272), (96, 33, 144), (96, 25, 1040), (144, 40, 16),
                                   (144, 33, 4096), (96, 64, 8208), (144, 40, 16400)])
def test_gradients(kt, F, K, B):
    m, p, x, t, rng = setup(kt, F, K, B, 11)
    compare(m, p, x, t, rng.integers(0, len(x), size=B).astype(np.int32))


def test_batches_of_both_ends_on_one_handle(kt):
    """Three Adam steps of 8,208 rows and three of 16: the losses follow the oracle's, and
    the gradients afterwards are those of the parameters the handle then has."""
    m, p, x, t, rng = setup(kt, 96, 33, 8208, 5)
    opt = omlp.Adam(p)
    for B in (8208, 16):
        idx = rng.integers(0, len(x), size=3 * B).astype(np.int32)
        losses = m.train(idx, B)
        for s in range(3):
            b = idx[s * B:(s + 1) * B]
            oloss, g = omlp.loss_and_grads(p, x[b], t[b])
            # an update is at most the learning rate (1e-3) in either direction where a
            # gradient's sign is within rounding: far below a hundredth of the loss
            assert abs(losses[s] - oloss) <= 1e-2 * oloss, (B, s)
            opt.step(p, g)
        now = m.get_params()
        for B2 in (16, 1040):
            compare(m, now, x, t, rng.integers(0, len(x), size=B2).astype(np.int32))


@pytest.mark.parametrize("K", [1, 33, 64])
def test_predictions_of_three_feature_chunks(kt, K):
    m, p, x, t, rng = setup(kt, 144, K, 16, 7)
    raw = rng.integers(0, 1 << 32, size=700).astype(np.int64)
    got = m.predict(raw)
    dig = np.stack(np.unravel_index(raw, RADICES[144]), axis=1)
    ref, _ = omlp.forward(p, omlp.features([list(range(1, 17))] * 8, dig))
    ref = ref * np.linspace(1.0, 50.0, K).astype(np.float32)
    scale = np.max(np.abs(ref), axis=0) + 1e-6
    assert np.all(np.max(np.abs(got - ref), axis=0) <= 5e-3 * scale)
