"""Batches with more MLP groups than the step has branches, one network's searches in
more than one group, and tree searches beside them, against the searches on their own."""
import numpy as np
import pytest

import workloads as W
from test_gpu_batch import kt, run_batch, run_single  # noqa: F401
from workloads.synth import SyntheticGPU
from workloads.trees import random_model

pytestmark = pytest.mark.gpu


def make(kt, stream=None):  # noqa: F811
    from paper_2102_05297_gb300 import fit
    out, keep = [], []
    for si, (radices, mlps, trees) in enumerate([((16, 9, 7), 10, 1), ((5, 5), 1, 0), ((16, 16, 5, 4), 2, 2),
                                                 ((3, 11, 13), 3, 1), ((2, 9, 16, 3), 1, 3)]):
        d = W.SpaceDesc("g", ["p%d" % j for j in range(len(radices))],
                        [list(range(1, r + 1)) for r in radices], [])
        K = [16, 32, 40, 32, 16][si]
        roles = W.layout(K)
        gpu = SyntheticGPU(d, roles, seed=si)
        sp = kt.Space.from_desc(d)
        mlp = kt.Mlp(sp, roles, gpu.counter_ranges(), max_batch=16)
        p = fit.init_mlp(mlp.F, K, seed=si)
        p["b4"] = np.full(K, 0.5, np.float32)
        mlp.set_params(p)
        mm, tm = kt.Model.from_mlp(mlp), kt.Model(sp, random_model(d.radices, roles, depth=6 + si, seed=si))
        keep += [sp, mlp, mm, tm]
        for r in range(mlps + trees):
            model = mm if r < mlps else tm
            out.append((d, gpu, sp, model, kt.Search(sp, model, k=3, seed=50 * si + r, search_id=r, stream=stream)))
    return out, keep


@pytest.mark.parametrize("own_stream", [False, True])
def test_groups_match_single_searches(kt, own_stream):  # noqa: F811
    import torch
    stream = torch.cuda.Stream() if own_stream else None
    a, keep_a = make(kt, stream)
    b, keep_b = make(kt)
    assert run_batch(kt, a, 4, 3, stream=stream) == run_single(b, 4, 3)
