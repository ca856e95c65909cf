"""Steps of several searches on one GPU: the default grids of spaces below 2^18
configurations pick what the four kernels pick, whichever entry point steps, and the
steps of searches on different streams run side by side."""
import time

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


def setup(kt, radices, K, depth, seed):
    desc = W.SpaceDesc("f", ["p%d" % j for j in range(len(radices))],
                       [list(range(1, r + 1)) for r in radices], [])
    roles = W.layout(K)
    sp = kt.Space.from_desc(desc)
    m = kt.Model(sp, random_model(desc.radices, roles, depth=depth, seed=seed))
    c = SyntheticGPU(desc, roles, seed=seed).evaluate(np.zeros((1, len(radices)), dtype=np.int64))[0][0]
    return sp, m, c


# configurations: 4,368 (16 CTAs), 77,760 and 78,000 (76 and 77 of 1,024), 155,520 and
# more (148)
@pytest.mark.parametrize("select", ["sample", "topk"])
@pytest.mark.parametrize("radices", [(14, 13, 12, 2), (15, 16, 12, 9, 3), (13, 15, 16, 5, 5), (15, 16, 12, 9, 6),
                                     (13, 15, 16, 5, 10), (15, 16, 12, 9, 9), (13, 15, 16, 12, 7)])
def test_both_entry_points_in_turn(kt, radices, select):
    import torch
    sp, m, c = setup(kt, radices, 16, 7, 3)
    sel = kt.KTUNE_SELECT_TOPK if select == "topk" else kt.KTUNE_SELECT_SAMPLE
    runs = []
    for shape in (0, None):
        st = torch.cuda.Stream()
        s = kt.Search(sp, m, k=9, seed=4, select=sel, stream=st)
        if shape is not None:
            s.set_fused(shape)
        raw = torch.zeros(9, dtype=torch.int64, device="cuda")
        sc = torch.zeros(9, device="cuda")
        torch.cuda.synchronize()
        seq = []
        for i in range(6):
            if i in (1, 2, 4):
                s.step_device(c, 9, raw.data_ptr(), sc.data_ptr(), stream=st)
                torch.cuda.synchronize()
                seq.append((raw.tolist(), sc.tolist()))
            else:
                r, x = s.step(c)
                seq.append((r.tolist(), x.tolist()))
            if i == 3 and shape is None:
                s.set_fused(1)           # every SM from here on
        runs.append(seq)
        s.close()
    assert runs[0] == runs[1]


@pytest.mark.parametrize("radices", [(16, 16, 16, 10), (16, 16, 16, 10, 4)])   # 40,960 and 163,840
def test_steps_on_different_streams_overlap(kt, radices):
    """Eight searches enqueued on eight streams take less than half of eight times one
    (0.9 of it with a CTA on every SM; a quarter here)."""
    import torch
    n = 8
    e = []
    for i in range(n):
        sp, m, c = setup(kt, radices, 32, 12, 3)
        st = torch.cuda.Stream()
        e.append((kt.Search(sp, m, k=5, seed=i, stream=st), c, st, torch.zeros(5, dtype=torch.int64, device="cuda"),
                  torch.zeros(5, device="cuda"), sp, m))
    torch.cuda.synchronize()

    def go(searches, rounds):
        t = time.perf_counter()
        for _ in range(rounds):
            for s, c, st, raw, sc, _, _ in searches:
                s.step_device(c, 5, raw.data_ptr(), sc.data_ptr(), stream=st)
        torch.cuda.synchronize()
        return time.perf_counter() - t

    go(e, 3)
    one = min(go(e[:1], 30) for _ in range(4))
    all_ = min(go(e, 30) for _ in range(4))
    assert all_ < 0.5 * n * one, (all_, one)
