"""Draws of more than one look-ahead round (16 of them) over spaces of many and of few
sub-tiles against the oracle, in the persistent and the four-kernel step, and
neighbourhood draws on both sides of the size up to which they stay in registers."""
import numpy as np
import pytest

import workloads as W
from oracle import nbr as onbr, space as ospace
from oracle.search import OracleSearch
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


def make(radices, K, depth, seed):
    desc = W.SpaceDesc("d", ["p%d" % j for j in range(len(radices))],
                       [list(range(1, r + 1)) for r in radices], [])
    roles = W.layout(K)
    return desc, random_model(desc.radices, roles, depth=depth, seed=seed), SyntheticGPU(desc, roles, seed=seed)


# 5,120 configurations (5 sub-tiles: most draws share one) and 156,000 (153)
@pytest.mark.parametrize("radices", [(16, 16, 5, 4), (13, 15, 16, 5, 10)])
@pytest.mark.parametrize("k,gamma", [(17, -0.25), (33, 0.5), (64, -0.05)])
@pytest.mark.parametrize("shape", [0, None])
def test_draws_match_oracle(kt, radices, k, gamma, shape):
    desc, model, gpu = make(radices, 16, 7, 2)
    sp = kt.Space.from_desc(desc)
    s = kt.Search(sp, kt.Model(sp, model), k=k, seed=6, gamma=gamma)
    if shape is not None:
        s.set_fused(shape)
    o = OracleSearch(desc, model, k=k, seed=6, gamma=gamma)
    assert s.current() == o.cprof_raw
    for step in range(4):
        c = gpu.evaluate(ospace.decode(desc.radices, [s.current()]))[0][0]
        if step == 2:
            c = c * 0              # no bottleneck: all configurations weigh the same
        raw, sc = s.step(c)
        o_raw, o_sc = o.step(c)
        assert list(raw) == o_raw
        np.testing.assert_array_equal(sc, np.float32(o_sc))
        rt = np.arange(k, 0, -1, dtype=float)
        s.report(rt)
        o.report(list(rt))


# 3,829 candidates (eight per thread), 4,011 and 4,102 (the compacted list): the oracle
# holds c_profile and its neighbours alone, which is all that these steps look at
@pytest.mark.parametrize("last,n_cand", [(5, 3829), (7, 4011), (8, 4102)])
def test_neighbourhood_draws_around_4096_candidates(kt, last, n_cand):
    radices = [16] * 6 + [last]
    desc, model, gpu = make(radices, 16, 9, 4)
    sp = kt.Space.from_desc(desc)
    k = 64
    s = kt.Search(sp, kt.Model(sp, model), k=k, seed=3)
    s.set_neighbourhood(2)
    cp = s.current()
    dig = ospace.decode(radices, [cp])[0]
    strides = np.array([int(np.prod(radices[j + 1:], dtype=np.int64)) for j in range(len(radices))])
    near = onbr.neighbour_digits(radices, dig, 2)
    assert len(near) == n_cand
    o = onbr.NbrSearch(desc, model, radius=2, k=k, seed=3, valid=np.sort(np.append(near @ strides, cp)))
    o.cprof = int(np.searchsorted(o.valid, cp))
    o.evaluated[:] = False
    o.evaluated[o.cprof] = True
    c = gpu.evaluate(dig[None])[0][0]
    for _ in range(3):
        raw, sc = s.step(c)
        o_raw, o_sc = o.step(c)
        assert list(raw) == o_raw
        np.testing.assert_array_equal(sc, np.float32(o_sc))
