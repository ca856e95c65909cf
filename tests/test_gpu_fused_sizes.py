"""Steps of materialised spaces by their default shape and by every persistent
kernel, against the four kernels: every score, weight and pick, where a CTA's
share of the space ends at or next to 1, 2, 4, 5 and 8 configurations per thread."""
import numpy as np
import pytest

import workloads as W
from workloads.synth import SyntheticGPU
from workloads.trees import random_model

pytestmark = pytest.mark.gpu

# configurations (per CTA of 152): 4,368 (28), 77,760 (511.6), 78,000 (513.2), 155,520
# (1,023.2), 156,000 (1,026.3), 233,280 (1,534.7), 311,040 (2,046.3), 312,000
# (2,052.6), 388,800 (2,557.9), 622,080 (4,092.6), 624,000 (4,105.3: two chunks)
SIZES = [(14, 13, 12, 2), (15, 16, 12, 9, 3), (13, 15, 16, 5, 5), (15, 16, 12, 9, 6),
         (13, 15, 16, 5, 10), (15, 16, 12, 9, 9), (15, 16, 12, 9, 12), (13, 15, 16, 10, 10),
         (15, 16, 12, 9, 15), (15, 16, 12, 9, 12, 2), (13, 15, 16, 10, 10, 2)]


@pytest.fixture(scope="module")
def kt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2102_05297_gb300 import ktune
    return ktune


@pytest.mark.parametrize("select", ["sample", "topk"])
@pytest.mark.parametrize("i", range(len(SIZES)))
def test_default_and_persistent_steps_match_four_kernels(kt, i, select):
    import torch
    radices = SIZES[i]
    desc = W.SpaceDesc("f", ["p%d" % j for j in range(len(radices))],
                       [list(range(1, r + 1)) for r in radices], [])
    roles = W.layout(16)
    gpu = SyntheticGPU(desc, roles, seed=4)
    sp = kt.Space.from_desc(desc)
    n = sp.count()[0]
    assert n == int(np.prod(radices))
    m = kt.Model(sp, random_model(desc.radices, roles, depth=(8, 12, 5)[i % 3], seed=i))
    sel = kt.KTUNE_SELECT_TOPK if select == "topk" else kt.KTUNE_SELECT_SAMPLE
    runs = []
    for shape in (0, None, 1, 2, 3):
        s = kt.Search(sp, m, k=7, seed=9, select=sel)
        if shape is not None:
            s.set_fused(shape)
        seq = []
        for _ in range(2):
            c = gpu.evaluate(np.stack(np.unravel_index([s.current()], radices), axis=1))[0][0]
            raw, sc = s.step(c)
            s.report(np.arange(1, len(raw) + 1, dtype=np.float64))
            sd = torch.zeros(n, device="cuda")
            wd = torch.zeros(n, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            s.scores_device(0, n, sd.data_ptr(), wd.data_ptr() if select == "sample" else 0)
            torch.cuda.synchronize()
            seq.append((np.array(raw), np.array(sc), sd.cpu().numpy(), wd.cpu().numpy()))
        runs.append(seq)
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            for x, y in zip(a, b):
                np.testing.assert_array_equal(x, y)


def test_timed_steps_of_small_spaces_keep_four_kernels(kt):
    """Per-kernel times come from the four kernels until a shape is asked for; the
    steps are the same with and without them."""
    radices = SIZES[1]
    desc = W.SpaceDesc("f", ["p%d" % j for j in range(len(radices))], [list(range(1, r + 1)) for r in radices], [])
    roles = W.layout(16)
    gpu = SyntheticGPU(desc, roles, seed=4)
    sp = kt.Space.from_desc(desc)
    m = kt.Model(sp, random_model(desc.radices, roles, depth=6, seed=1))
    runs = []
    for timed in (False, True):
        s = kt.Search(sp, m, k=3, seed=2)
        s.set_timing(timed)
        c = gpu.evaluate(np.stack(np.unravel_index([s.current()], radices), axis=1))[0][0]
        runs.append([list(x) for x in s.step(c)])
        assert s.stats().n_kernels == (4 if timed else 0)
    assert runs[0] == runs[1]
    s.set_fused(2)
    s.step(c)
    assert s.stats().n_kernels == 1
