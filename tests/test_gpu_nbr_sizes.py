"""Neighbourhood-restricted steps against the oracle where a thread holds one,
two or three candidates, where the draws take up to every candidate, and with
more counters than a warp has lanes."""
import pytest

import workloads as W
from test_gpu_nbr import drive, kt  # noqa: F401
from workloads.synth import SyntheticGPU
from workloads.trees import random_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radices,K,depth,radius,k", [
    ((2, 2), 16, 3, 1, 64),               # 2 candidates
    ((3, 1, 5), 16, 4, 2, 64),            # a parameter with one value; 14 candidates, all taken
    ((16, 16, 8), 40, 11, 2, 64),         # 502: one per thread
    ((16, 16, 16, 5), 40, 6, 2, 33),      # 904: two
    ((16, 16, 16, 16), 32, 12, 2, 7)])    # 1,410: three
def test_draws_match_oracle(kt, radices, K, depth, radius, k):  # noqa: F811
    desc = W.SpaceDesc("n", ["p%d" % j for j in range(len(radices))],
                       [list(range(1, r + 1)) for r in radices], [])
    roles = W.layout(K)
    model = random_model(desc.radices, roles, depth=depth, seed=K)
    gpu = SyntheticGPU(desc, roles, seed=radius)
    _, _, n = drive(kt, desc, model, gpu, radius, "sample", steps=3, k=k, seed=2)
    assert n >= 1
