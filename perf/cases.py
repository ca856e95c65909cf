"""The work that users of this framework have it do, as cases that can be timed.

A tuner creates a space, fits or trains a counter model on a sample of
profiles, and then steps a search: the counters of the last profiled
configuration go in, the next configurations to run come out.  The cases below
are those calls at the sizes of the repository's own spaces and models (the
spaces under workloads/spaces, the counter layouts of 16, 32 and 40 counters,
depth-8 and depth-12 trees, the 3 x 256 MLP, batches of 4096 training rows), and
generated spaces without constraints between them.  Counters and profile
samples come from the seeded synthetic GPU of workloads/synth.py.

The models are fitted quickly, not well: trees by the best of a few random
splits per node, the MLP's output layer by least squares on random hidden
layers.  Their predictions have the counters' scale and depend on the
parameters, which is what a step's work and its scores depend on.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_2102_05297_gb300 import fit
from paper_2102_05297_gb300 import ktune as kt
from workloads.synth import SyntheticGPU, add_noise

HIDDEN = 256
INST_REACTION, CORES = 0.7, 1000.0
# valid configurations of the frozen spaces (tests/golden/space_counts.json)
N_VALID = {"tiny_block_tile": 1824, "batch_0": 316096, "batch_1": 988416, "batch_2": 3456,
           "batch_3": 17100, "batch_4": 149760, "batch_5": 127488, "batch_6": 46656,
           "batch_7": 162816, "mid_12p": 2257920, "large_16p": 19525632}
BATCH_K = [16, 32, 40, 16, 32, 40, 16, 32]     # counters of the eight batch spaces


# ---------------------------------------------------------------------------
def listed():
    return [
        # A whole tuning run over a small space, as the paper's benchmarks have
        # (a few thousand configurations): the search is created, stepped 40
        # times with the runtimes of its picks reported, and closed.
        dict(name="session_tiny", kind="session", space="tiny_block_tile", K=16, depth=8, k=5,
             steps=40, stream=False),
        # One step over a space of ordinary size, the program on its own stream.
        dict(name="step_trees_160k", kind="step", model="tree", space="batch_7", K=32, depth=12,
             k=5, select="sample", otf=False, mode="plain", stream=True),
        # The same over millions of configurations, with depth-12 trees for 32
        # counters: the workload of the repository's benchmark.
        dict(name="step_trees_2m", kind="step", model="tree", space="mid_12p", K=32, depth=12,
             k=5, select="sample", otf=False, mode="plain", stream=True),
        # A space too large to keep: decoded from its 113M raw indices in every
        # step, the 16 best taken.
        dict(name="step_otf_20m_top16", kind="step", model="tree", space="large_16p", K=40,
             depth=12, k=16, select="topk", otf=True, mode="plain", stream=False),
        # The paper's other model, least-squares polynomials per subspace; the
        # program looks at every score and weight.
        dict(name="step_lsq_2m", kind="step", model="lsq", space="mid_12p", K=32, depth=0, k=5,
             select="sample", otf=False, mode="plain", read=True, stream=True),
        # A long search that keeps the trees' predictions between steps.
        dict(name="step_cached_2m", kind="step", model="tree", space="mid_12p", K=32, depth=12,
             k=5, select="sample", otf=False, mode="cached", stream=True),
        # Local search: only configurations at distance 1 or 2 are scored, so
        # the step is all latency.
        dict(name="step_nbr2", kind="step", model="tree", space="mid_12p", K=32, depth=12, k=5,
             select="sample", otf=False, mode="nbr2", stream=True),
        # The learned model: every step predicts the space with the network
        # (scores and weights read as well).
        dict(name="step_mlp_2m", kind="step", model="mlp", space="mid_12p", K=32, depth=0, k=5,
             select="sample", otf=False, mode="plain", read=True, stream=True),
        # A tuning service: 64 searches over eight spaces (trees and MLPs in
        # turn, eight searches per space), one batched step for all.
        dict(name="batch_64", kind="batch", spaces=8, per_space=8, depth=12, k=5, stream=True),
        # Training of the MLP on collected profiles.
        dict(name="train_mlp_4096", kind="train", space="mid_12p", K=32, rows=40000, batch=4096,
             steps=16, stream=True),
        # Predicted counters of a range of the space, for checks of the model
        # and for a user's own ranking; odd start and length.
        dict(name="predict_mlp_2m", kind="predict", model="mlp", space="large_16p", K=40, depth=0,
             first=1234567, count=2000003),
        # Start of a program: the space enumerated and its configurations read
        # (the seed gives the order in which the program lists the parameters).
        dict(name="create_41m_raw", kind="create", space="mid_12p", otf=False),
    ]


def _flat(rng, lo, hi):
    """A space without constraints of lo to hi configurations, its size spread
    over the logarithm, its digits within one 32-bit word."""
    while True:
        target, radices, n, bits = math.exp(rng.uniform(math.log(lo), math.log(hi))), [], 1, 0
        while n < target and len(radices) < 14:
            r = rng.choice([2, 2, 3, 4, 5, 6, 7, 8, 11, 16])
            radices.append(r)
            n *= r
            bits += max(1, (r - 1).bit_length())
        if lo <= n <= hi and bits <= 32:
            return "flat:" + ".".join(map(str, radices))


def draw(rng):
    kind = rng.choice(["session", "step", "step", "step", "step", "step", "batch", "train",
                       "predict", "create"])
    K = rng.choice([16, 32, 40])
    if kind == "session":
        return dict(kind=kind, space=rng.choice(["tiny_block_tile", "batch_2", "batch_3",
                                                 _flat(rng, 1500, 20000)]),
                    K=K, depth=rng.randint(6, 12), k=rng.randint(1, 8), steps=rng.randint(10, 40),
                    stream=rng.random() < 0.5)
    if kind == "step":
        model = rng.choice(["tree", "tree", "tree", "lsq", "mlp"])
        space = rng.choice(["batch_0", "batch_1", "batch_4", "batch_5", "batch_6", "batch_7",
                            "mid_12p"] + [_flat(rng, 40000, 2200000) for _ in range(5)])
        c = dict(kind=kind, model=model, space=space, K=K, depth=rng.randint(7, 12),
                 k=rng.choice([1, 3, 5, 5, 8, 16, 33, 64]), select="sample", otf=False,
                 mode="plain", stream=rng.random() < 0.5)
        if model != "tree":
            c["depth"] = 0
            c["mode"] = rng.choice(["plain", "plain", "cached"])
        else:
            form = rng.choice(["plain", "plain", "topk", "otf", "otf_topk", "cached", "nbr1", "nbr2"])
            if form in ("otf", "otf_topk"):
                c["otf"] = True
                c["space"] = rng.choice([space, "large_16p"])
            if form in ("topk", "otf_topk"):
                c["select"] = "topk"
            if form in ("cached", "nbr1", "nbr2"):
                c["mode"] = form
            if form == "nbr1":
                c["k"] = rng.randint(1, 5)
        c["read"] = c["select"] == "sample" and not c["mode"].startswith("nbr") and rng.random() < 0.3
        return c
    if kind == "batch":
        return dict(kind=kind, spaces=rng.randint(1, 8), per_space=rng.randint(1, 8),
                    depth=rng.randint(7, 12), k=rng.randint(1, 8), stream=rng.random() < 0.5)
    if kind == "train":
        return dict(kind=kind, space=rng.choice(["mid_12p", "batch_1", "batch_7", "large_16p"]), K=K,
                    rows=rng.randint(3000, 40000),
                    batch=16 * int(round(math.exp(rng.uniform(math.log(8), math.log(256))))),
                    steps=rng.randint(4, 16), stream=rng.random() < 0.5)
    if kind == "predict":
        space = rng.choice(["batch_1", "batch_6", "mid_12p", "large_16p"])
        count = int(math.exp(rng.uniform(math.log(200), math.log(min(2000000, N_VALID[space] - 1)))))
        return dict(kind=kind, model=rng.choice(["mlp", "mlp", "tree", "lsq"]) if space != "batch_6" else "mlp",
                    space=space, K=K, depth=rng.randint(7, 12),
                    first=rng.randint(0, N_VALID[space] - count), count=count)
    return dict(kind=kind, space=rng.choice(["batch_0", "batch_1", "batch_3", "batch_7", "mid_12p",
                                             _flat(rng, 2000, 2200000)]), otf=rng.random() < 0.3)


# ---------------------------------------------------------------------------
def _desc(name):
    if name == "tiny_block_tile":
        return W.space_tiny_block_tile()
    if name.startswith("flat:"):
        r = [int(x) for x in name[5:].split(".")]
        return W.SpaceDesc(name, ["p%d" % j for j in range(len(r))],
                           [[1 << i if n <= 8 else i + 1 for i in range(n)] for n in r], [])
    return W.load_space(name)


def _reordered(desc, rng):
    """The same space with its parameters in another order."""
    order = rng.permutation(desc.n_params)          # new parameter i is the old order[i]
    where = np.argsort(order)
    code, i = list(desc.bytecode), 0
    while i < len(code):
        if code[i] == W.OP_VAL:
            code[i + 1] = int(where[code[i + 1]])
        i += 3 if code[i] == W.OP_CONST64 else 2 if code[i] in W.OPS_WITH_ARG else 1
    return W.SpaceDesc(desc.name, [desc.param_names[j] for j in order],
                       [desc.values[j] for j in order], code)


def _n_valid(name):
    return N_VALID[name] if name in N_VALID else _desc(name).n_raw


def _digits_of(radices, raw):
    raw = np.array(raw, dtype=np.int64)
    out = np.empty((len(raw), len(radices)), dtype=np.int64)
    for j in range(len(radices) - 1, -1, -1):
        out[:, j] = raw % radices[j]
        raw //= radices[j]
    return out


def _sample_raw(sp, desc, n, rng):
    """Raw indices of n configurations spread over TS (materialised spaces)."""
    total = sp.count()[0]
    runs = min(n, 64)
    width = min(total, -(-n // runs))
    starts = rng.integers(0, total - width + 1, size=runs)
    return np.concatenate([sp.valid_raw(int(a), width) for a in starts])[:n]


def _forest(digits, Y, depth, rng):
    """One tree per counter: per node the best of three random splits."""
    X = np.asarray(digits, dtype=np.int64)
    trees = []
    for c in range(Y.shape[1]):
        y = np.asarray(Y[:, c], dtype=np.float64)
        feature, threshold, left, right, value = [[-1]], [[0]], [[-1]], [[-1]], [[y.mean()]]
        base, size = 0, 1                     # ids of the level's nodes: base .. base + size
        rows, node = np.arange(len(X)), np.zeros(len(X), dtype=np.int64)
        for _ in range(depth):
            cnt = np.bincount(node, minlength=size)
            tot = np.bincount(node, weights=y[rows], minlength=size)
            first = np.concatenate([[0], np.cumsum(cnt)[:-1]])
            order = np.argsort(node, kind="stable")
            best, bf, bt = np.full(size, -np.inf), np.zeros(size, np.int64), np.zeros(size, np.int64)
            for _ in range(3):
                f = rng.integers(0, X.shape[1], size=size)
                some = rows[order[first + (rng.random(size) * cnt).astype(np.int64)]]
                t = np.maximum(X[some, f] - 1, 0)
                go = X[rows, f[node]] > t[node]
                nr = np.bincount(node, weights=go, minlength=size)
                sr = np.bincount(node, weights=go * y[rows], minlength=size)
                with np.errstate(divide="ignore", invalid="ignore"):
                    g = sr * sr / nr + (tot - sr) ** 2 / (cnt - nr)
                g = np.where((nr > 0) & (nr < cnt), g, -np.inf)
                better = g > best
                best, bf, bt = np.where(better, g, best), np.where(better, f, bf), np.where(better, t, bt)
            split = best > -np.inf
            if not split.any():
                break
            ids = np.cumsum(split) - 1         # rank among the level's inner nodes
            feature[-1] = np.where(split, bf, -1)
            threshold[-1] = np.where(split, bt, 0)
            left[-1] = np.where(split, base + size + 2 * ids, -1)
            right[-1] = np.where(split, base + size + 2 * ids + 1, -1)
            keep = split[node]
            rows, node = rows[keep], node[keep]
            node = 2 * ids[node] + (X[rows, bf[node]] > bt[node])
            base, size = base + size, 2 * int(split.sum())
            n2 = np.bincount(node, minlength=size)
            value.append(np.bincount(node, weights=y[rows], minlength=size) / n2)
            feature.append(np.full(size, -1))
            threshold.append(np.zeros(size))
            left.append(np.full(size, -1))
            right.append(np.full(size, -1))
        cat = lambda parts, dt: np.concatenate([np.asarray(p) for p in parts]).astype(dt)  # noqa: E731
        trees.append({"feature": cat(feature, np.int32), "threshold": cat(threshold, np.int32),
                      "left": cat(left, np.int32), "right": cat(right, np.int32),
                      "value": cat(value, np.float32)})
    return trees


def _u(values):
    out = []
    for v in values:
        l = np.log2(1.0 + np.asarray(v, dtype=np.float64))
        out.append(np.zeros(len(v)) if l.max() == l.min() else
                   2.0 * (l - l.min()) / (l.max() - l.min()) - 1.0)
    return out


def _features(values, digits, F):
    """One-hot digits, then u per parameter, zero-padded to F (float64, on the GPU)."""
    d = torch.as_tensor(digits, device="cuda")
    n, P = d.shape
    x = torch.zeros((n, F), dtype=torch.float64, device="cuda")
    off = 0
    for j, v in enumerate(values):
        x[torch.arange(n, device="cuda"), off + d[:, j]] = 1.0
        off += len(v)
    for j, u in enumerate(_u(values)):
        x[:, off + j] = torch.as_tensor(u, device="cuda")[d[:, j]]
    return x


def _forward(p, x):
    for i in (1, 2, 3):
        x = torch.nn.functional.gelu(x @ p["W%d" % i].T + p["b%d" % i])
    return x @ p["W4"].T + p["b4"]


def _mlp_params(values, F, K, digits, Y, ranges, seed):
    """Random hidden layers and an output layer fitted by least squares."""
    p = fit.init_mlp(F, K, seed=seed)
    for i in (1, 2, 3):
        p["W%d" % i] *= np.float32(1.6)      # keeps the activations' spread through the layers
    q = {k: torch.as_tensor(v, dtype=torch.float64, device="cuda") for k, v in p.items()}
    h = _features(values, digits, F)
    for i in (1, 2, 3):
        h = torch.nn.functional.gelu(h @ q["W%d" % i].T + q["b%d" % i])
    h = torch.cat([h, torch.ones((len(h), 1), dtype=torch.float64, device="cuda")], 1)
    t = torch.as_tensor(Y / ranges, dtype=torch.float64, device="cuda")
    ridge = 1e-3 * len(h) * torch.eye(h.shape[1], dtype=torch.float64, device="cuda")
    w = np.linalg.solve((h.T @ h + ridge).cpu().numpy(), (h.T @ t).cpu().numpy())
    p["W4"], p["b4"] = w[:-1].T.astype(np.float32), w[-1].astype(np.float32)
    return p


def _sample(sp, desc, case, rng):
    """Digits of a profile sample: valid configurations, or any raw indices of
    a space that is not materialised."""
    if case.get("otf"):
        return np.stack([rng.integers(0, r, size=4096) for r in desc.radices], axis=1)
    return _digits_of(desc.radices, _sample_raw(sp, desc, min(4096, sp.count()[0]), rng))


def _fit(kind, desc, roles, gpu, digits, depth, seed):
    """The model as plain arrays (no handle), from noisy profiles."""
    Y = add_noise(gpu.evaluate(digits)[0], seed, 0.02)
    if kind == "tree":
        return {"roles": roles, "trees": _forest(digits, Y, depth, np.random.default_rng(seed))}
    if kind == "lsq":
        return fit.fit_lsq(desc.values, digits, Y, roles)
    F = -(-(sum(desc.radices) + desc.n_params) // 16) * 16
    return _mlp_params(desc.values, F, len(roles), digits, Y, gpu.counter_ranges(), seed)


def _model(sp, kind, plain, roles, gpu, stream):
    if kind != "mlp":
        return kt.Model(sp, plain)
    mlp = kt.Mlp(sp, roles, gpu.counter_ranges(), max_batch=4096, stream=stream)
    mlp.set_params(plain)
    return kt.Model.from_mlp(mlp)


def _new_search(st):
    c = st["case"]
    s = kt.Search(st["space"], st["model"], k=c["k"], seed=st["seed"], stream=st["stream"],
                  select=kt.KTUNE_SELECT_TOPK if c["select"] == "topk" else kt.KTUNE_SELECT_SAMPLE)
    if c["mode"] == "cached":
        s.set_cached(True)
    elif c["mode"] in ("nbr1", "nbr2"):
        s.set_neighbourhood(int(c["mode"][3:]))
    return s


def _profiles(sp, desc, case, gpu, rng, n, search):
    """Configurations that a search's c_profile may be, and their counters."""
    if case["otf"]:
        raw = []
        while len(raw) < n:
            r = int(rng.integers(0, desc.n_raw))
            try:
                search.set_profile(r)
                raw.append(r)
            except kt.KtuneError:            # violates the constraints
                pass
    else:
        raw = [int(r) for r in _sample_raw(sp, desc, n, rng)]
    counters = gpu.evaluate(_digits_of(desc.radices, raw))[0]
    return list(zip(raw, counters))


def prepare(case, seed):
    rng = np.random.default_rng([seed, 77])
    stream = torch.cuda.Stream() if case.get("stream") else None
    st = {"case": case, "seed": seed, "stream": stream, "i": 0}
    if case["kind"] == "create":
        st["desc"] = _reordered(_desc(case["space"]), rng)
        return st
    if case["kind"] == "batch":
        return _prepare_batch(st, case, seed, rng)
    desc = _desc(case["space"])
    roles = W.layout(case["K"])
    gpu = SyntheticGPU(desc, roles, seed=seed)
    sp = kt.Space.from_desc(desc, flags=kt.KTUNE_ON_THE_FLY if case.get("otf") else kt.KTUNE_MATERIALISE)
    st.update(space=sp, desc=desc)
    if case["kind"] == "train":
        raw = _sample_raw(sp, desc, case["rows"], rng)
        mlp = kt.Mlp(sp, roles, gpu.counter_ranges(), max_batch=4096, stream=stream)
        mlp.set_params(fit.init_mlp(mlp.F, case["K"], seed=seed))
        mlp.set_data(raw, add_noise(gpu.evaluate(_digits_of(desc.radices, raw))[0], seed, 0.02))
        idx = rng.integers(0, len(raw), size=case["steps"] * case["batch"]).astype(np.int32)
        st.update(mlp=mlp, idx=idx)
        return st
    kind = case.get("model", "tree")
    plain = _fit(kind, desc, roles, gpu, _sample(sp, desc, case, rng), case["depth"], seed)
    st["model"] = _model(sp, kind, plain, roles, gpu, stream)
    if case["kind"] == "session":
        st["raw"] = sp.valid_raw()
        st["counters"], st["runtime"] = gpu.evaluate(sp.valid_digits())
    elif case["kind"] == "predict":
        st["out"] = torch.empty((case["count"], case["K"]), dtype=torch.float32, device="cuda")
    else:
        st["search"] = _new_search(st)
        n = 1024 if case["mode"].startswith("nbr") else 64
        st["profiles"] = _profiles(sp, desc, case, gpu, rng, n, st["search"])
        st["left"] = sp.count()[0] - 1
        if case.get("read"):
            n = sp.count()[0]
            st["scores"] = torch.empty(n, dtype=torch.float32, device="cuda")
            st["weights"] = torch.empty(n, dtype=torch.int32, device="cuda")
    return st


def _prepare_batch(st, case, seed, rng):
    searches, counters, keep = [], [], []
    for i in range(case["spaces"]):
        desc, roles = _desc("batch_%d" % i), W.layout(BATCH_K[i])
        gpu = SyntheticGPU(desc, roles, seed=seed + i)
        sp = kt.Space.from_desc(desc)
        kind = "mlp" if i % 2 else "tree"
        plain = _fit(kind, desc, roles, gpu, _sample(sp, desc, case, rng), case["depth"], seed + i)
        m = _model(sp, kind, plain, roles, gpu, st["stream"])
        keep.append((sp, m))
        for r in range(case["per_space"]):
            s = kt.Search(sp, m, k=case["k"], seed=seed + 10 * i + r, search_id=r, stream=st["stream"])
            searches.append(s)
            counters.append(gpu.evaluate(_digits_of(desc.radices, [s.current()]))[0][0])
    st.update(keep=keep, searches=searches, counters=counters,
              batch=kt.Batch(searches, stream=st["stream"]))
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        if state["left"] < case["k"]:        # the space is used up: the search starts over
            state["search"].close()
            state["search"] = _new_search(state)
            state["left"] = state["space"].count()[0] - 1
        raw, counters = state["profiles"][state["i"] % len(state["profiles"])]
        state["i"] += 1
        state["search"].set_profile(raw)
        try:
            picks, scores = state["search"].step(counters, case["k"])
        except kt.KtuneError:
            if not case["mode"].startswith("nbr"):
                raise
            return []                        # nothing left around this configuration
        state["left"] -= len(picks)
        if case.get("read"):
            state["search"].scores_device(0, len(state["scores"]), state["scores"].data_ptr(),
                                          state["weights"].data_ptr(), state["stream"])
            return [picks, scores, state["scores"], state["weights"]]
        return [picks, scores]
    if kind == "session":
        s = kt.Search(state["space"], state["model"], k=case["k"], seed=state["seed"],
                      stream=state["stream"])
        picks, scores = [], []
        for _ in range(case["steps"]):
            at = int(np.searchsorted(state["raw"], s.current()))
            raw, sc = s.step(state["counters"][at])
            s.report(state["runtime"][np.searchsorted(state["raw"], raw)])
            picks.append(raw)
            scores.append(sc)
        last = s.current()
        s.close()
        return [np.concatenate(picks), np.concatenate(scores), last]
    if kind == "batch":
        out = state["batch"].step(state["counters"], case["k"])
        return [np.concatenate([raw for raw, _ in out]), np.concatenate([sc for _, sc in out])]
    if kind == "train":
        losses = state["mlp"].train(state["idx"], case["batch"])
        return {"losses": losses, **state["mlp"].get_params()}
    if kind == "predict":
        m = state["model"]
        m = m.mlp if case["model"] == "mlp" else m
        m.predict_device(case["first"], case["count"], state["out"].data_ptr(),
                         torch.cuda.current_stream())
        return state["out"]
    sp = kt.Space.from_desc(state["desc"], flags=kt.KTUNE_ON_THE_FLY if case["otf"] else kt.KTUNE_MATERIALISE)
    out = list(sp.count())
    if not case["otf"]:
        out.append(sp.valid_raw())
    sp.close()
    return out


# ---------------------------------------------------------------------------
# Counters with a reaction, about, of a profile of the synthetic GPU.
ACTIVE = 9


def _mlp_flops(radices, K):
    # per configuration: the one-hot part of the first layer is one row per parameter
    return 2.0 * (2 * len(radices) * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN * K)


def _step_work(n, case, desc, model, depth, K):
    """One whole-space step: a digit word and an evaluated bit per configuration,
    the model, and the operations of the active counters."""
    bytes_ = n * (4 + 1 / 8)
    if case.get("otf"):
        bytes_ = n / 8
    if model == "mlp":
        F = -(-(sum(desc.radices) + desc.n_params) // 16) * 16
        weights = 2 * HIDDEN * (F + 2 * HIDDEN + K)
        flops = n * (_mlp_flops(desc.radices, K) + 5 * ACTIVE)
    elif model == "lsq":
        m = sum(r > 2 for r in desc.radices)
        T = 1 + 2 * m + m * (m - 1) // 2
        weights = 4 * T * ACTIVE * (1 << sum(r == 2 for r in desc.radices))
        flops = n * ACTIVE * (2 * T + 5)
    else:
        weights = ACTIVE * 5 * (1 << depth)
        flops = n * ACTIVE * (depth + 1)      # a visit counted as one operation
    if case.get("mode") == "cached":
        bytes_ = n * ACTIVE * (2 if model == "tree" else 4) + n / 8
        flops = n * ACTIVE * (1 if model == "tree" else 5)
    return bytes_ + weights, flops + 10 * n   # normalisation, weight and their sum


def work(case):
    if case["kind"] == "batch":
        b = f = 0.0
        for i in range(case["spaces"]):
            desc = _desc("batch_%d" % i)
            x, y = _step_work(_n_valid("batch_%d" % i), case, desc, "mlp" if i % 2 else "tree",
                              case["depth"], BATCH_K[i])
            b, f = b + case["per_space"] * x, f + (1 if i % 2 else case["per_space"]) * y
        return {"bytes": b, "flops": f}
    desc, n = _desc(case["space"]), _n_valid(case["space"])
    if case["kind"] == "create":
        return {"bytes": 8.0 * n if not case["otf"] else 8.0, "flops": 10.0 * desc.n_raw}
    if case["kind"] == "train":
        B, S = case["batch"], case["steps"]
        weights = HIDDEN * (sum(desc.radices) + desc.n_params + 2 * HIDDEN + case["K"])
        return {"bytes": float(S * B * (4 + 8 + 4 * case["K"]) + 2 * 12 * weights),
                "flops": 3.0 * S * B * _mlp_flops(desc.radices, case["K"])}
    if case["kind"] == "predict":
        c, K = case["count"], case["K"]
        if case["model"] == "mlp":
            f = c * _mlp_flops(desc.radices, K)
        elif case["model"] == "lsq":
            m = sum(r > 2 for r in desc.radices)
            f = 2.0 * c * K * (1 + 2 * m + m * (m - 1) // 2)
        else:
            f = float(c * K * case["depth"])
        return {"bytes": c * (8.0 + 4 * K), "flops": f}
    model = case.get("model", "tree")
    if case["kind"] == "step" and case["mode"].startswith("nbr"):
        r = [x - 1 for x in desc.radices]
        c = sum(r)
        if case["mode"] == "nbr2":
            c += (sum(r) ** 2 - sum(x * x for x in r)) // 2
        return {"bytes": c * 16.0 + ACTIVE * 5.0 * (1 << case["depth"]),
                "flops": float(c * (ACTIVE * (case["depth"] + 1) + 10))}
    b, f = _step_work(n, case, desc, model, case["depth"], case["K"])
    if case.get("read"):
        b += 8.0 * n
    k = case["steps"] if case["kind"] == "session" else 1
    return {"bytes": k * b, "flops": k * f}


# ---------------------------------------------------------------------------
# What the calls compute, in 64 bits, by plain numpy and torch.  A search's draws
# are decisions taken on 32-bit weights, so the scores of what it draws have no
# value of their own in 64 bits: trees' scores of a whole space, top-k scores,
# predictions and training do.  (A polynomial's or a network's predictions take
# both signs, so Eq. score's denominator comes arbitrarily near to zero and its
# score has no stable value either; their predictions have.)
def _holds(code, val):
    """Whether the constraint program holds: val[j] are int64 tensors."""
    ok, st, i = None, [], 0

    def div(a, b):
        safe = torch.where(b == 0, torch.ones_like(b), b)
        q = torch.div(a, safe, rounding_mode="trunc")
        return torch.where(b == 0, torch.zeros_like(q), q), torch.where(b == 0, torch.zeros_like(q), a - q * safe)

    one = torch.ones_like(val[0])
    while i < len(code):
        op = code[i]
        i += 1
        if op in (W.OP_VAL, W.OP_CONST):
            st.append(val[code[i]] if op == W.OP_VAL else one * code[i])
            i += 1
        elif op == W.OP_CONST64:
            st.append(one * ((code[i + 1] << 32) | (code[i] & 0xFFFFFFFF)))
            i += 2
        elif op == W.OP_REQUIRE:
            c = st.pop() != 0
            ok = c if ok is None else ok & c
        elif op == W.OP_NOT:
            st.append((st.pop() == 0).long())
        else:
            b, a = st.pop(), st.pop()
            st.append({W.OP_ADD: lambda: a + b, W.OP_SUB: lambda: a - b, W.OP_MUL: lambda: a * b,
                       W.OP_DIV: lambda: div(a, b)[0], W.OP_MOD: lambda: div(a, b)[1],
                       W.OP_EQ: lambda: (a == b).long(), W.OP_NE: lambda: (a != b).long(),
                       W.OP_LT: lambda: (a < b).long(), W.OP_LE: lambda: (a <= b).long(),
                       W.OP_GT: lambda: (a > b).long(), W.OP_GE: lambda: (a >= b).long(),
                       W.OP_AND: lambda: ((a != 0) & (b != 0)).long(),
                       W.OP_OR: lambda: ((a != 0) | (b != 0)).long()}[op]())
    return ok if ok is not None else torch.ones_like(one, dtype=torch.bool)


def _valid_chunks(desc, chunk=1 << 23):
    """Digits [n, P] (int64, on the GPU) of the valid configurations, in raw order."""
    for lo in range(0, desc.n_raw, chunk):
        raw = torch.arange(lo, min(desc.n_raw, lo + chunk), device="cuda")
        dig = []
        for r in reversed(desc.radices):
            dig.append(raw % r)
            raw = raw // r
        dig.reverse()
        val = [torch.as_tensor(v, device="cuda")[d] for v, d in zip(desc.values, dig)]
        ok = _holds(desc.bytecode, val)
        yield torch.stack([d[ok] for d in dig], 1)


def _delta(roles, counters):
    """Bottlenecks and the reaction to them (Section 3.4 of the method), float64."""
    pc = {}
    for r, v in zip(roles, counters):
        pc.setdefault(W.ROLE_NAMES[r], float(v))
    neutral = {"SM_E": 100.0, "WARP_E": 100.0, "WARP_NP_E": 100.0}
    g = lambda x: pc.get(x, neutral.get(x, 0.0))  # noqa: E731
    unit = lambda x: min(1.0, max(0.0, x))        # noqa: E731
    out = {}
    for a, b, u in (("DRAM_RT", "DRAM_WT", "DRAM_U"), ("L2_RT", "L2_WT", "L2_U"),
                    ("SHR_LT", "SHR_WT", "SHR_U")):
        for x in (a, b):
            out[x] = -unit(g(x) / (g(a) + g(b)) * g(u) / 100.0) if g(a) + g(b) > 0 else 0.0
    out["TEX_RWT"] = -unit(g("TEX_U") / 100.0)
    out["LOC_O"] = -unit(g("LOC_O") / 100.0 * max(g("DRAM_U"), g("L2_U"), g("TEX_U")) / 100.0)
    fitted = 32.0 * g("INST_EXE") * (100.0 / (g("WARP_E") or 100.0)) * (100.0 / (g("WARP_NP_E") or 100.0))
    react = lambda b: 0.0 if b <= INST_REACTION else -(b - INST_REACTION) / (1.0 - INST_REACTION)  # noqa: E731
    most = 0.0
    for x in ("F32", "F64", "INT", "MISC", "LDST", "CONT", "BCONV"):
        part = g("INST_" + x) / fitted if fitted > 0 else 0.0
        most = max(most, part)
        out["INST_" + x] = react(unit(part * min(1.0, g("INST_ISSUE_U") / 50.0)))
    out["INST_ISSUE_U"] = react(unit(most * (100.0 - g("INST_ISSUE_U")) / 100.0))
    out["SM_E"] = unit((100.0 - g("SM_E")) / 100.0)
    out["GLOBAL"] = unit((5.0 * CORES - pc["GLOBAL"]) / (5.0 * CORES)) if "GLOBAL" in pc else 0.0
    delta, seen = np.zeros(len(roles)), set()
    for i, r in enumerate(roles):
        name = W.ROLE_NAMES[r]
        if name in out and name not in seen:
            delta[i] = out[name]
            seen.add(name)
    return delta


def _walk(tree, dig):
    t = {k: torch.as_tensor(v, device="cuda").long() for k, v in tree.items() if k != "value"}
    at = torch.zeros(len(dig), dtype=torch.int64, device="cuda")
    while True:
        f = t["feature"][at]
        if not bool((f >= 0).any()):
            return torch.as_tensor(tree["value"], device="cuda").double()[at]
        d = dig.gather(1, f.clamp(min=0)[:, None])[:, 0]
        nxt = torch.where(d > t["threshold"][at], t["right"][at], t["left"][at])
        at = torch.where(f >= 0, nxt, at)


def _lsq(values, coef, dig):
    u = _u(values)
    regs = [j for j, v in enumerate(values) if len(v) > 2]
    U = [torch.as_tensor(u[j], device="cuda")[dig[:, j]] for j in regs]
    sub = torch.zeros(len(dig), dtype=torch.int64, device="cuda")
    for j, v in enumerate(values):
        if len(v) == 2:
            sub = sub * 2 + dig[:, j]
    X = torch.stack([torch.ones(len(dig), dtype=torch.float64, device="cuda")] + U + [x * x for x in U] +
                    [U[a] * U[b] for a in range(len(U)) for b in range(a + 1, len(U))], 1)
    c = torch.as_tensor(coef, device="cuda").double()
    out = torch.empty((len(dig), c.shape[1]), dtype=torch.float64, device="cuda")
    for s in range(c.shape[0]):
        rows = torch.nonzero(sub == s)[:, 0]
        out[rows] = X[rows] @ c[s].T
    return out


def _exact_predict(case, desc, kind, plain, ranges):
    out, seen = [], 0
    if kind == "mlp":
        p = {k: torch.as_tensor(v, device="cuda").double() for k, v in plain.items()}
        F, scale = plain["W1"].shape[1], torch.as_tensor(ranges, device="cuda").float().double()
    for dig in _valid_chunks(desc):
        lo, hi = max(case["first"], seen), min(case["first"] + case["count"], seen + len(dig))
        if lo < hi:
            for d in torch.split(dig[lo - seen:hi - seen], 1 << 18):
                if kind == "mlp":
                    y = _forward(p, _features(desc.values, d, F)) * scale
                elif kind == "lsq":
                    y = _lsq(desc.values, plain["coef"], d)
                else:
                    y = torch.stack([_walk(t, d) for t in plain["trees"]], 1)
                out.append(y)
        seen += len(dig)
    return torch.cat(out)


def _exact_scores(desc, roles, plain, raw, counters):
    """Eq. score of every configuration with the trees, in TS order, by chunks."""
    delta = _delta(roles, counters)
    me = torch.as_tensor(_digits_of(desc.radices, [raw]), device="cuda")
    on = [(float(delta[i]), float(_walk(t, me)[0]), t) for i, t in enumerate(plain["trees"]) if delta[i]]
    for dig in _valid_chunks(desc):
        s = torch.zeros(len(dig), dtype=torch.float64, device="cuda")
        for d, mine, tree in on:
            if mine:
                a = _walk(tree, dig)
                s += torch.where(a != 0, d * (a - mine) / (a + mine), torch.zeros_like(a))
        yield s


def _exact_train(case, desc, gpu, raw, idx, seed):
    p = fit.init_mlp(-(-(sum(desc.radices) + desc.n_params) // 16) * 16, case["K"], seed=seed)
    p = {k: torch.as_tensor(v, device="cuda").double().requires_grad_() for k, v in p.items()}
    dig = _digits_of(desc.radices, raw)
    Y = add_noise(gpu.evaluate(dig)[0], seed, 0.02)
    x = _features(desc.values, dig, p["W1"].shape[1])
    t = torch.as_tensor(Y / gpu.counter_ranges(), device="cuda").double()
    opt = torch.optim.Adam(list(p.values()), lr=1e-3)
    losses = []
    for rows in torch.as_tensor(idx, device="cuda").long().split(case["batch"]):
        opt.zero_grad()
        loss = ((_forward(p, x[rows]) - t[rows]) ** 2).mean()
        loss.backward()
        opt.step()
        losses.append(loss.detach())
    return {"losses": torch.stack(losses), **{k: v.detach() for k, v in p.items()}}


def exact(case, seed):
    topk = case["kind"] == "step" and case["select"] == "topk"
    read = case.get("read") and case["model"] == "tree"
    if case["kind"] not in ("predict", "train") and not topk and not read:
        return None
    if topk and _n_valid(case["space"]) < 100000:
        return None          # the first, already evaluated configuration may be among the best
    # the inputs as prepare() makes them
    rng = np.random.default_rng([seed, 77])
    desc = _desc(case["space"])
    roles = W.layout(case["K"])
    gpu = SyntheticGPU(desc, roles, seed=seed)
    sp = kt.Space.from_desc(desc, flags=kt.KTUNE_ON_THE_FLY if case.get("otf") else kt.KTUNE_MATERIALISE)
    if case["kind"] == "train":
        raw = _sample_raw(sp, desc, case["rows"], rng)
        idx = rng.integers(0, len(raw), size=case["steps"] * case["batch"]).astype(np.int32)
        return _exact_train(case, desc, gpu, raw, idx, seed)
    kind = case["model"]
    plain = _fit(kind, desc, roles, gpu, _sample(sp, desc, case, rng), case["depth"], seed)
    if case["kind"] == "predict":
        return _exact_predict(case, desc, kind, plain, gpu.counter_ranges())
    search = kt.Search(sp, _model(sp, kind, plain, roles, gpu, None), k=case["k"], seed=seed)
    raw, counters = _profiles(sp, desc, case, gpu, rng, 64, search)[0]
    scores = _exact_scores(desc, roles, plain, raw, counters)
    if topk:
        best = torch.empty(0, dtype=torch.float64, device="cuda")
        for s in scores:
            best = torch.cat([best, s]).sort(descending=True)[0][:case["k"]]
        return [None, best]
    return [None, None, torch.cat(list(scores)), None]
