"""The work that a user of this library has it do, as measurable cases.

An autotuner's explorer screens batches of candidate configurations with a
validity ensemble V and a performance ensemble P, keeps the best k, reranks
them with a deeper ensemble A, moves annealing chains through the knob space
and materialises decoded knob spaces.  Every case goes through the public
Python entry points of `paper_2411_10764_gb300.mlt` on buffers that such a
program holds on the GPU.

A case is one of seven kinds:
  screen          stored features, fp32 or binary16 tables, balanced trees or
                  unbalanced ones, with or without missing values
  screen_decoded  candidates of a knob space, features built by the library
  until           batched accumulation that stops at a target count
  sa_step         one annealing move of many chains
  rerank          model A over the kept candidates
  decode          a knob space's option indices and features, materialised
The ensembles are a function of the case alone (an explorer loads them once
and screens many batches with them); the candidates come from the seed.
"""
from __future__ import annotations

import math
import statistics

import numpy as np
import torch

from paper_2411_10764_gb300 import mlt
from paper_2411_10764_gb300 import workloads as W

_SAMPLE_ROWS = 4096  # rows whose quantiles are the stored cases' thresholds
_LEAF_SIGMA = 0.1


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def _screen(name, n, F, vt, vd, pt, pd, thr, k, survival=0.4, knobs=8, knob_values=11, sigma=1.0, zeros=0.0,
            nan=0.0, dup=0.0, p_split=1.0, v_split=1.0, zipf=False, half=False):
    """n candidates of F features (`knobs` small-integer columns, the rest
    lognormal); V has vt trees of depth vd, P pt of depth pd; a node below the
    root splits with probability *_split."""
    return dict(name=name, kind="screen", n=n, F=F, vt=vt, vd=vd, pt=pt, pd=pd, thr=thr, k=k, survival=survival,
                knobs=knobs, knob_values=knob_values, sigma=sigma, zeros=zeros, nan=nan, dup=dup, p_split=p_split,
                v_split=v_split, zipf=zipf, half=half)


def _decoded(kind, n, F=96, vt=300, vd=10, pt=600, pd=10, thr=0.5, k=1024, **more):
    return dict(kind=kind, n=n, F=F, vt=vt, vd=vd, pt=pt, pd=pd, thr=thr, k=k, survival=0.45, v_split=1.0,
                p_split=1.0, **more)


def listed():
    return [
        # the smallest batch of the benchmark: launches and hand-offs count
        _screen("tiny-4096x32", 4096, 32, 50, 6, 100, 6, 0.5, 64, knob_values=7),
        # the paper's own model sizes (300 rounds, V depth 5, P depth 14) over
        # one explorer batch of an odd size, keeping (alpha + 1) N = 20
        _screen("paper-models-20011x47", 20011, 47, 300, 5, 300, 14, 0.5, 20, p_split=0.75, knobs=12),
        # the benchmark's gemm tuning batch
        _screen("gemm-65536x64", 65536, 64, 200, 8, 400, 8, 0.5, 128, knobs=12, sigma=1.5, zeros=0.1),
        # the same batch through half tables
        _screen("gemm-half-65536x64", 65536, 64, 200, 8, 400, 8, 0.5, 128, knobs=12, sigma=1.5, zeros=0.1, half=True),
        # rows that no vector load is aligned to, a few missing values, V and
        # P of different depths
        _screen("ragged-300007x101", 300007, 101, 300, 7, 500, 9, 0.55, 300, nan=0.02, dup=0.01, knobs=16),
        # a large simulated-annealing batch
        _screen("sa-batch-1048576x128", 1 << 20, 128, 500, 8, 1000, 8, 0.6, 512, survival=0.3, knobs=24),
        # deep unbalanced ensembles, skewed split features, many missing values
        _screen("skewed-nan-4194304x256", 1 << 22, 256, 1000, 12, 2000, 12, 0.5, 2048, survival=0.55, knobs=16,
                nan=0.3, dup=0.05, v_split=0.9, p_split=0.9, zipf=True),
        # all but a little of the conv2d knob space (16,777,216 candidates),
        # decoded by the library
        dict(_decoded("screen_decoded", 16_700_000), name="conv2d-16700000x96"),
        # accumulate batches until 7,693 candidates are kept
        dict(_screen("", 65536, 64, 200, 8, 400, 8, 0.5, 128, knobs=12, sigma=1.5, zeros=0.1), kind="until",
             batch=8192, target=7693, name="until-65536x64"),
        # one annealing move of 131,072 chains over the conv2d space
        dict(_decoded("sa_step", 131072, temperature=1.0), name="sa-step-131072x96"),
        # model A (300 trees, depth 14) over the 128 kept candidates
        dict(kind="rerank", n=65536, F=64, m=128, n_final=64, at=300, ad=14, a_split=0.75, knobs=12, knob_values=11,
             sigma=1.5, zeros=0.1, nan=0.0, dup=0.0, name="rerank-128of65536x64"),
        # materialise a quarter of the conv2d space
        dict(kind="decode", n=1 << 22, F=96, name="decode-4194304x96"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_stored(rng, most_visits):
    """Sizes of a stored batch whose V and P visits stay below most_visits."""
    deep = rng.random() < 0.3
    if deep:
        vd, pd = rng.choice([(5, 14), (11, 12), (12, 12), (8, 13)])
        v_split, p_split = (1.0 if vd <= 10 else rng.uniform(0.7, 0.9)), rng.uniform(0.7, 0.9)
        path = 7.2
    else:
        vd = rng.randint(4, 10)
        pd = vd if rng.random() < 0.6 else rng.randint(4, 10)
        v_split = p_split = 1.0
        path = max(vd, pd)
    F = _log_int(rng, 16, 256)
    vt, pt = _log_int(rng, 50, 1000), _log_int(rng, 100, 1000)
    top = min(4e6, most_visits / ((vt + 0.5 * pt) * path), 1.5e9 / F)
    n = _log_int(rng, 1000, max(2000, top))
    nan = rng.choice([0.0, 0.0, 0.0, 0.02, 0.3])
    return _screen("", n, F, vt, vd, pt, pd, rng.choice([0.5, 0.5, 0.6]), min(_log_int(rng, 16, 2048), n),
                   survival=rng.uniform(0.2, 0.55), knobs=min(F // 2, rng.randint(4, 24)), sigma=rng.uniform(0.7, 1.5),
                   zeros=rng.choice([0.0, 0.1]), nan=nan, dup=rng.choice([0.0, 0.05]), v_split=v_split,
                   p_split=p_split, zipf=rng.random() < 0.2)


def draw(rng):
    kind = rng.choice(["screen"] * 6 + ["half", "screen_decoded", "screen_decoded", "until", "sa_step", "rerank",
                                        "decode"])
    if kind in ("screen", "half", "until"):
        c = _draw_stored(rng, 2e10)
        if kind == "half":
            c.update(half=True, vd=min(c["vd"], 10), pd=min(c["pd"], 10))
        if kind == "until":
            c.update(kind="until", n=min(c["n"], 400000))
            c.update(batch=max(500, c["n"] // rng.randint(3, 12)))
            c.update(target=max(1, int(c["n"] * rng.uniform(0.05, 0.4))), k=min(c["k"], c["n"]))
        del c["name"]
        return c
    if kind == "screen_decoded":
        n = _log_int(rng, 4000, 1 << 23)
        return _decoded("screen_decoded", n, F=rng.randint(64, 128), vt=_log_int(rng, 100, 300), vd=rng.randint(6, 10),
                        pt=_log_int(rng, 200, 600), pd=rng.randint(6, 10), k=min(_log_int(rng, 64, 1024), n))
    if kind == "sa_step":
        return _decoded("sa_step", _log_int(rng, 128, 1 << 20), F=rng.randint(64, 128), vt=_log_int(rng, 100, 300),
                        vd=rng.randint(6, 10), pt=_log_int(rng, 200, 600), pd=rng.randint(6, 10),
                        temperature=rng.uniform(0.1, 2.0))
    if kind == "rerank":
        m = _log_int(rng, 20, 2048)
        F = _log_int(rng, 16, 256)
        return dict(kind="rerank", n=_log_int(rng, 5000, 300000), F=F, m=m, n_final=max(1, m // 2),
                    at=_log_int(rng, 100, 500), ad=rng.choice([8, 12, 14, 14]), a_split=rng.uniform(0.7, 0.85),
                    knobs=F // 4, knob_values=11, sigma=1.0, zeros=0.0, nan=rng.choice([0.0, 0.1]), dup=0.0)
    return dict(kind="decode", n=_log_int(rng, 10000, 1 << 22), F=rng.randint(64, 128))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _features(c, seed, n):
    """[n][F] fp32 on the GPU: small-integer knob columns, then lognormal
    ones, with exact zeros, missing values and duplicate rows as asked."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
    x = torch.empty((n, c["F"]), dtype=torch.float32, device="cuda")
    x.normal_(generator=g).mul_(c["sigma"]).exp_()
    kn = c["knobs"]
    if kn:
        x[:, :kn] = torch.randint(0, c["knob_values"], (n, kn), generator=g, device="cuda").to(torch.float32)
    step = max(1, (1 << 28) // c["F"])
    for a in range(0, n, step):
        y = x[a:a + step]
        if c["zeros"]:
            h = y[:, kn:]
            h.masked_fill_(torch.rand(h.shape, generator=g, device="cuda") < c["zeros"], 0.0)
        if c["nan"]:
            y.masked_fill_(torch.rand(y.shape, generator=g, device="cuda") < c["nan"], float("nan"))
    d = int(c["dup"] * n)
    if d:
        dst = torch.randperm(n, generator=g, device="cuda")[:d]
        src = torch.randint(0, n, (d,), generator=g, device="cuda")
        x[dst] = x[src]
    return x


class _Quantiles:
    """Thresholds drawn from the order statistics of a sample's columns."""

    def __init__(self, sample):
        self.sorted = np.sort(sample, axis=0).T.copy()  # NaN last
        self.count = np.sum(~np.isnan(sample), axis=0)

    def draw(self, rng, f):
        at = np.floor(rng.random(f.size) * np.maximum(self.count[f] - 1, 0)).astype(np.int64)
        return np.where(self.count[f] > 0, self.sorted[f, at], 0.0).astype(np.float32)


class _Ranges:
    """Thresholds inside the decoded features' value ranges, half of them
    whole numbers (log-uniform over wide positive ranges)."""

    def __init__(self, ranges):
        self.lo = np.array([r[0] for r in ranges])
        self.hi = np.array([r[1] for r in ranges])

    def draw(self, rng, f):
        lo, hi = self.lo[f], self.hi[f]
        u = rng.random(f.size)
        a, b = np.log(np.maximum(lo, 1e-30)), np.log(np.maximum(hi, 1e-30))
        t = np.where((lo > 0) & (hi > 64 * lo), np.exp(a + u * (b - a)), lo + u * (hi - lo))
        return np.where(rng.random(f.size) < 0.5, np.round(t), t).astype(np.float32)


def _ensemble(key, F, trees, depth, split_prob, thresholds, mean, zipf):
    """Random ensemble in the library's heap-order node layout."""
    rng = np.random.default_rng(np.random.SeedSequence(key))
    slots = (2 << depth) - 1
    nodes = np.zeros((trees, slots), dtype=W.NODE_DTYPE)
    split = np.zeros((trees, slots), dtype=bool)
    exists = np.zeros((trees, slots), dtype=bool)
    exists[:, 0] = True
    for d in range(depth):
        a, b = (1 << d) - 1, (2 << d) - 1
        split[:, a:b] = exists[:, a:b]
        if d and split_prob < 1.0:
            split[:, a:b] &= rng.random((trees, b - a), dtype=np.float32) < split_prob
        exists[:, 2 * a + 1:2 * b + 1] = np.repeat(split[:, a:b], 2, axis=1)
    leaf = exists & ~split
    n_split = int(split.sum())
    if zipf:
        p = 1.0 / np.arange(1, F + 1) ** 1.2
        f = rng.permutation(F)[np.searchsorted(np.cumsum(p / p.sum()), rng.random(n_split)).clip(0, F - 1)]
    else:
        f = rng.integers(0, F, n_split)
    nodes["feature"] = W.UNUSED
    nodes["feature"][split] = f
    nodes["value"][split] = thresholds.draw(rng, f)
    nodes["default_left"][split] = rng.integers(0, 2, n_split)
    nodes["feature"][leaf] = W.LEAF
    nodes["value"][leaf] = (mean + _LEAF_SIGMA * rng.standard_normal(int(leaf.sum()))).astype(np.float32)
    return nodes.reshape(-1)


def _leaf_mean(trees, thr, survival):
    """V's leaf mean: about `survival` of the candidates clear the cut."""
    z = statistics.NormalDist().inv_cdf(1.0 - survival)
    return (math.log(thr / (1.0 - thr)) - _LEAF_SIGMA * math.sqrt(trees) * z) / trees


_models = {}  # the models of the last case prepared: {key: (decoder, {slot: (nodes, trees, depth)})}
_loaded = [None]  # key of the models the library holds


def _key(c):
    """What the case's ensembles depend on: everything but the batch."""
    batch = ("name", "n", "k", "batch", "target", "temperature", "m", "n_final")
    return repr(sorted((f, v) for f, v in c.items() if f not in batch))


def _models_of(c):
    key = _key(c)
    if key not in _models:
        F, dec = c["F"], None
        if c["kind"] in ("screen_decoded", "sa_step", "decode"):
            dec = W.conv2d_decoder(1, F)
        slots = {}
        if c["kind"] != "decode":
            th = _Ranges(dec.ranges) if dec else _Quantiles(_features(c, 77, _SAMPLE_ROWS).cpu().numpy())
            zipf = c.get("zipf", False)
            if c["kind"] == "rerank":
                slots[mlt.MLT_MODEL_A] = (_ensemble([5, F], F, c["at"], c["ad"], c["a_split"], th, 0.0, zipf), c["at"],
                                          c["ad"])
            else:
                mean = _leaf_mean(c["vt"], c["thr"], c["survival"])
                slots[mlt.MLT_MODEL_V] = (_ensemble([3, F], F, c["vt"], c["vd"], c["v_split"], th, mean, zipf), c["vt"],
                                          c["vd"])
                slots[mlt.MLT_MODEL_P] = (_ensemble([4, F], F, c["pt"], c["pd"], c["p_split"], th, 0.0, zipf), c["pt"],
                                          c["pd"])
        _models.clear()
        _models[key] = (dec, slots)
    return _models[key]


def _load(c):
    """The case's ensembles in the library (they stay there while batches of
    the same task come and go)."""
    key = _key(c)
    if _loaded[0] == key:
        return
    _, slots = _models_of(c)
    if slots:
        mlt.set_num_features(c["F"])
    for slot, (nodes, trees, depth) in slots.items():
        (mlt.load_ensemble_f16 if c.get("half") else mlt.load_ensemble)(slot, nodes, trees, depth)
    _loaded[0] = key


def _first(c, seed, space):
    """Where a decoded batch begins: enumerations go on from batch to batch."""
    return int(np.random.default_rng(seed).integers(0, space - c["n"] + 1))


def prepare(case, seed):
    dec, _ = _models_of(case)
    _load(case)
    s = {"case": case, "key": _key(case), "dec": dec}
    kind = case["kind"]
    if kind in ("screen", "until", "rerank"):
        s["x"] = _features(case, seed, case["n"])
    if kind == "rerank":
        g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62) + 1)
        s["cand"] = torch.randperm(case["n"], generator=g, device="cuda")[: case["m"]].contiguous()
    if kind in ("screen_decoded", "decode"):
        s["first"] = _first(case, seed, dec.space)
    if kind == "sa_step":
        g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
        n = case["n"]
        s["parent"] = torch.randint(0, dec.space, (n,), generator=g, device="cuda")
        s["score"] = torch.empty(n, device="cuda").normal_(generator=g) * 2.0
        s["knob"] = torch.randint(0, 1 << 31, (n,), generator=g, device="cuda").to(torch.int32)
        s["digit"] = torch.randint(0, 1 << 31, (n,), generator=g, device="cuda").to(torch.int32)
        s["logu"] = torch.rand(n, generator=g, device="cuda").clamp_min(1e-30).log()
    return s


def run(state):
    c, dec = state["case"], state["dec"]
    if _loaded[0] != state["key"]:
        _load(c)  # another task's ensembles were loaded meanwhile
    kind = c["kind"]
    if kind == "screen":
        return mlt.screen(state["x"], c["thr"], c["k"])
    if kind == "until":
        # rows past the consumed prefix are not written, so only the kept
        # candidates and the counts are asked for
        _, _, topk, stats = mlt.screen_until(state["x"], c["batch"], c["target"], c["thr"], c["k"], with_outputs=False)
        return topk, stats
    if kind == "rerank":
        return mlt.rerank(state["x"], state["cand"], c["n_final"])
    if kind == "screen_decoded":
        return mlt.screen_decoded(dec.radices, dec.option_values, dec.program, state["first"], c["n"], c["thr"], c["k"])
    if kind == "sa_step":
        return mlt.sa_step(dec.radices, dec.option_values, dec.program, state["parent"], state["score"], state["knob"],
                           state["digit"], state["logu"], c["temperature"], c["thr"])
    return mlt.decode_knobs(dec.radices, dec.option_values, dec.program, state["first"], c["n"])


# ---------------------------------------------------------------------------
# What a pass cannot do without, and how exact it is
# ---------------------------------------------------------------------------

def _path(depth, split_prob):
    """Expected node tests on a path, and expected nodes of a tree."""
    p, length, nodes = 1.0, 0.0, 1.0
    for d in range(depth):
        p *= 1.0 if d == 0 else split_prob
        length += p
        nodes += p * (2 << d)
    return length, nodes


def work(case):
    """bytes: the features (or indices) in, the results out, each table's
    nodes (8 bytes: feature and value) once; flops: one compare per node test
    on a path and one add per leaf, for V over every candidate and for P over
    the expected survivors, one operation per decoded feature."""
    c, kind, F = case, case["kind"], case["F"]
    if kind == "rerank":
        length, nodes = _path(c["ad"], c["a_split"])
        return {"bytes": c["m"] * (4 * F + 12) + 8 * c["n_final"] + 8 * c["at"] * nodes,
                "flops": c["m"] * c["at"] * (length + 1)}
    if kind == "decode":
        return {"bytes": c["n"] * (4 * F + 8), "flops": c["n"] * F}
    vl, vn = _path(c["vd"], c["v_split"])
    pl, pn = _path(c["pd"], c["p_split"])
    n = c["n"]
    if kind == "until":
        n = min(n, -(-int(c["target"] / c["survival"]) // c["batch"]) * c["batch"])
    ops = n * (c["vt"] * (vl + 1) + c["survival"] * c["pt"] * (pl + 1))
    tables = 8 * (c["vt"] * vn + c["pt"] * pn)
    if kind == "sa_step":
        return {"bytes": n * (24 + 16) + tables, "flops": ops + n * F}
    if kind == "screen_decoded":
        return {"bytes": n * 8 + 8 * c["k"] + tables, "flops": ops + n * F}
    return {"bytes": n * (4 * F + (0 if kind == "until" else 8)) + 8 * c["k"] + tables, "flops": ops}


def tolerance(case):
    """Leaves are summed in fp32 in tree order and a score is documented to be
    that sum, so scores, decisions and indices have one right value; pvalid
    goes through the device's expf, which the library documents to 1e-6."""
    if case["kind"] in ("until", "rerank", "decode", "sa_step"):
        return "exact"
    return {"rel": 1e-6}


# ---------------------------------------------------------------------------
# The same results in 64 bits, without the library
# ---------------------------------------------------------------------------

_EXACT_MOST = 2.5e11  # node tests that torch does in about 20 seconds


def _program(dec, kv, dtype):
    """Feature columns of the knob values kv (a list of columns)."""
    cols = []

    def of(s, const):
        return torch.full_like(kv[0], float(const)) if s < 0 else kv[s] if s < len(kv) else cols[s - len(kv)]

    for o in dec.program:
        a, b = of(int(o["a"]), o["c"]), of(int(o["b"]), o["c"])
        op = int(o["op"])
        if op == W.OP_COPY:
            v = a
        elif op == W.OP_ILOG2:
            v = torch.where(a >= torch.finfo(torch.float32).tiny, torch.frexp(a)[1].to(dtype) - 1, torch.zeros_like(a))
        elif op == W.OP_ADD:
            v = a + b
        elif op == W.OP_SUB:
            v = a - b
        elif op == W.OP_MUL:
            v = a * b
        elif op == W.OP_DIV:
            v = a / b
        elif op == W.OP_CEILDIV:
            v = torch.ceil(a / b)
        elif op == W.OP_REM:
            v = a - b * torch.floor(a / b)
        elif op == W.OP_MIN:
            v = torch.where(b < a, b, a)
        elif op == W.OP_MAX:
            v = torch.where(b > a, b, a)
        elif op == W.OP_GT:
            v = (a > b).to(dtype)
        else:
            v = (a == b).to(dtype)
        cols.append(v)
    return cols


def _digits(dec, idx):
    out, rem = [], idx
    for r in dec.radices.tolist():
        out.append(rem % r)
        rem = rem // r
    return out


def _decode(dec, idx, dtype):
    """(digits, [F][n] features) of candidate indices."""
    digits, kv, off = _digits(dec, idx), [], 0
    opts = torch.from_numpy(dec.option_values.copy()).cuda().to(dtype)
    for d, r in zip(digits, dec.radices.tolist()):
        kv.append(opts[off + d])
        off += r
    return digits, torch.stack(_program(dec, kv, dtype))


def _margins(nodes, trees, depth, xt, rows=None):
    """Sums over trees of the leaf each candidate reaches, in float64; xt is
    [F][n], rows the candidates to walk (all if None)."""
    slots = (2 << depth) - 1
    nd = nodes.reshape(trees, slots)
    n = xt.shape[1] if rows is None else rows.numel()
    at = torch.arange(n, device="cuda", dtype=torch.int64) if rows is None else rows
    acc = torch.zeros(n, dtype=torch.float64, device="cuda")
    flat, width = xt.reshape(-1), xt.shape[1]
    for t in range(trees):
        feat = torch.from_numpy(nd["feature"][t].astype(np.int64)).cuda()
        val = torch.from_numpy(nd["value"][t].copy()).cuda()
        left = torch.from_numpy(nd["default_left"][t].astype(bool)).cuda()
        j = torch.zeros(n, dtype=torch.int64, device="cuda")
        for _ in range(depth):
            f = feat[j]
            x = flat[f.clamp_min(0) * width + at]
            right = torch.where(torch.isnan(x), ~left[j], x >= val[j])
            j = torch.where(f >= 0, 2 * j + 1 + right, j)
        acc += val[j].double()
    return acc


def _half(nodes):
    out = nodes.copy()
    out["value"] = nodes["value"].astype(np.float16).astype(np.float32)
    return out


def _best(perf, k, index):
    """Indices of the k best finite scores (score descending, index
    ascending), -1 padded."""
    order = torch.sort(perf, descending=True, stable=True).indices[:k]
    order = order[perf[order] > -math.inf]
    out = torch.full((k,), -1, dtype=torch.int64, device="cuda")
    out[: order.numel()] = index[order]
    return out


def _screened(c, slots, xt):
    vm = _margins(*slots[mlt.MLT_MODEL_V], xt)
    cut = math.log(c["thr"] / (1.0 - c["thr"])) if c["thr"] != 0.5 else 0.0
    rows = torch.nonzero(vm >= cut).reshape(-1)
    perf = torch.full_like(vm, -math.inf)
    perf[rows] = _margins(*slots[mlt.MLT_MODEL_P], xt, rows)
    return torch.sigmoid(vm), perf


def exact(case, seed):
    c, kind = case, case["kind"]
    if work(c)["flops"] > _EXACT_MOST:
        return None
    state = prepare(c, seed)
    dec, slots = _models_of(c)
    if c.get("half"):
        slots = {m: (_half(nodes), t, d) for m, (nodes, t, d) in slots.items()}
    if kind == "decode":
        idx = state["first"] + torch.arange(c["n"], device="cuda", dtype=torch.int64)
        digits, x = _decode(dec, idx, torch.float64)
        return torch.stack(digits, 1).to(torch.uint8), x.T.contiguous()
    if kind == "rerank":
        score = _margins(*slots[mlt.MLT_MODEL_A], state["x"].T.contiguous(), state["cand"])
        by_index = torch.sort(state["cand"]).indices
        return score, _best(score[by_index], c["n_final"], state["cand"][by_index])
    if kind in ("screen", "until"):
        x = state.pop("x")
        if c.get("half"):
            x = x.half().float()
        xt = x.T.contiguous()
        del x
        if kind == "screen":
            pv, pf = _screened(c, slots, xt)
            return pv, pf, _best(pf, c["k"], torch.arange(c["n"], device="cuda"))
        used = kept = batches = 0
        _, pf = _screened(c, slots, xt)
        while used < c["n"] and kept < c["target"]:
            used = min(c["n"], used + c["batch"])
            kept = int((pf[:used] > -math.inf).sum())
            batches += 1
        return _best(pf[:used], c["k"], torch.arange(used, device="cuda")), torch.tensor([used, kept, batches])
    if kind == "screen_decoded":
        idx = state["first"] + torch.arange(c["n"], device="cuda", dtype=torch.int64)
        pv, pf = _screened(c, slots, _decode(dec, idx, torch.float32)[1])
        return pv, pf, _best(pf, c["k"], idx)
    # sa_step: set one knob, screen the proposal, accept by Metropolis
    parent, place, prop = state["parent"], 1, torch.zeros_like(state["parent"])
    pick = state["knob"].long() % len(dec.radices)
    for j, (d, r) in enumerate(zip(_digits(dec, parent), dec.radices.tolist())):
        prop += torch.where(pick == j, state["digit"].long() % r, d) * place
        place *= r
    _, s = _screened(c, slots, _decode(dec, prop, torch.float32)[1])
    ok = (s > -math.inf) & (s - state["score"].double() >= c["temperature"] * state["logu"].double())
    return torch.where(ok, prop, parent), torch.where(ok, s, state["score"].double()), ok.to(torch.int32)
