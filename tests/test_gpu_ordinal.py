"""The ordinal walk against the oracle, bit for bit, where it can go wrong:
block and tile edges, every depth, odd and even feature counts, aligned and unaligned rows, missing values on both default
sides, values on and beside the thresholds, infinities, one threshold, a full
search tree, and the models it must refuse."""
import numpy as np
import pytest

import oracle as O
from paper_2411_10764_gb300 import mlt
from paper_2411_10764_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N0 = 16384


@pytest.fixture(autouse=True)
def _always_ordinal():
    """These models are smaller than the rule's, so the walk is asked for."""
    mlt.tune_ordinal(2)
    yield
    mlt.tune_ordinal(1)


def _trees(rng, F, trees, depth, pool, split=1.0):
    slots = (2 << depth) - 1
    nodes = np.zeros((trees, slots), dtype=W.NODE_DTYPE)
    nodes["feature"] = W.UNUSED
    exists = np.zeros((trees, slots), dtype=bool)
    exists[:, 0] = True
    for j in range(slots):
        inner = exists[:, j] & (j < (1 << depth) - 1) & ((rng.random(trees) < split) | (j == 0))
        f = rng.integers(0, F, trees)
        nodes["feature"][:, j] = np.where(inner, f, np.where(exists[:, j], W.LEAF, W.UNUSED))
        nodes["value"][:, j] = np.where(inner, pool[rng.integers(0, pool.size, trees)], rng.normal(0, 0.1, trees))
        nodes["default_left"][:, j] = rng.integers(0, 2, trees)
        if 2 * j + 2 < slots:
            exists[:, 2 * j + 1] = exists[:, 2 * j + 2] = inner
    return W.Ensemble(nodes.reshape(-1), trees, depth)


def _rows(rng, n, F, pool, nan, special=True):
    x = rng.normal(0, 1, (n, F)).astype(np.float32)
    on = rng.random((n, F)) < 0.3  # on a threshold, or one float beside it
    v = pool[rng.integers(0, pool.size, (n, F))]
    side = rng.integers(0, 3, (n, F))
    v = np.where(side == 0, v, np.where(side == 1, np.nextafter(v, np.float32(-np.inf)), np.nextafter(v, np.float32(np.inf))))
    x[on] = v[on]
    if special:
        for s in (np.inf, -np.inf, 0.0, -0.0, 1e-45, -1e-45, 3.4e38, -3.4028235e38):
            x[rng.integers(0, n, 40), rng.integers(0, F, 40)] = s
    x[rng.random((n, F)) < nan] = np.nan
    return x


def _pool(rng, m):
    p = np.unique(rng.normal(0, 1, 2 * m).astype(np.float32))
    rng.shuffle(p)
    return p[:m]


def _check(x, v, p, thr, k, half=False, launches=6, offset=0):
    import torch

    mlt.set_num_features(x.shape[1])
    load = mlt.load_ensemble_f16 if half else mlt.load_ensemble
    load(mlt.MLT_MODEL_V, v.nodes, v.n_trees, v.depth)
    load(mlt.MLT_MODEL_P, p.nodes, p.n_trees, p.depth)
    flat = torch.empty(x.size + offset, dtype=torch.float32, device="cuda")
    flat[offset:] = torch.from_numpy(x.reshape(-1)).cuda()
    before = mlt.kernel_launches()
    pv, pf, tk = mlt.screen(flat[offset:].view(x.shape), thr, k)
    mlt.sync_status()
    assert mlt.kernel_launches() - before == launches
    if half:
        x, v, p = O.round_half(x), O.half_ensemble(v), O.half_ensemble(p)
    opv, opf, valid, _ = O.screen_rows(x, v, p, thr)
    otk, _ = O.topk(opf, valid, k)
    assert np.array_equal(pf.cpu().numpy().view(np.uint32), opf.view(np.uint32))
    assert np.array_equal(tk.cpu().numpy(), otk)
    # the oracle's own pvalid tolerance (device expf against host exp)
    assert np.all(np.abs(pv.cpu().numpy().astype(np.float64) - opv) <= 1e-6 * np.maximum(np.abs(opv), 1e-30))


@pytest.mark.parametrize("depth", range(1, 11))
def test_depths(depth):
    rng = np.random.default_rng(depth)
    F = 5 + depth % 3
    pool = _pool(rng, 50)
    trees = 16 * F // depth + 5  # ends on every remainder of the tree padding
    x = _rows(rng, N0 + 31 * depth, F, pool, nan=0.1 if depth % 2 else 0.0)
    _check(x, _trees(rng, F, trees, depth, pool), _trees(rng, F, trees + 2, depth, pool, split=0.8), 0.5, 100)


@pytest.mark.parametrize("F,offset", [(1, 0), (2, 0), (3, 1), (4, 0), (4, 1), (8, 0), (33, 0), (64, 0), (101, 2)])
def test_feature_counts_and_alignment(F, offset):
    rng = np.random.default_rng(F + offset)
    pool = _pool(rng, 300)
    trees = 16 * F // 6 + 1
    x = _rows(rng, N0 + 1, F, pool, nan=0.02)
    _check(x, _trees(rng, F, trees, 6, pool), _trees(rng, F, trees, 6, pool), 0.5, 64, offset=offset)


@pytest.mark.parametrize("n", [N0, N0 + 31, N0 + 33, 20000, 65537])
@pytest.mark.parametrize("keep", ["none", "few", "all"])
def test_sizes_and_survivors(n, keep):
    rng = np.random.default_rng(n)
    pool = _pool(rng, 7)
    x = _rows(rng, n, 3, pool, nan=0.0)
    v = _trees(rng, 3, 12, 5, pool)
    leaves = v.nodes["feature"] == W.LEAF
    v.nodes["value"][leaves] += {"none": -2.0, "few": -0.05, "all": 2.0}[keep]
    _check(x, v, _trees(rng, 3, 12, 5, pool), 0.5, 200)


@pytest.mark.parametrize("m", [1, 2, 3, 4, 255, 256, 4096, 8191])
def test_distinct_thresholds(m):
    """Search trees of every fullness; one feature holds m thresholds."""
    rng = np.random.default_rng(m)
    pool = np.sort(_pool(rng, m))
    trees, depth = max(4, -(-m // 511) + 1), 9
    v = _trees(rng, 2, trees, depth, pool)
    split = np.flatnonzero(v.nodes["feature"] >= 0)
    v.nodes["feature"][split[:m]] = 0
    v.nodes["value"][split[:m]] = pool
    v.nodes["feature"][split[m:]] = 1
    x = _rows(rng, N0 + 5, 2, pool, nan=0.05)
    _check(x, v, _trees(rng, 2, 8, 5, pool), 0.5, 64)


def test_too_many_thresholds_keep_the_fp32_walk():
    rng = np.random.default_rng(5)
    pool = _pool(rng, 8192)
    v = _trees(rng, 1, 17, 9, pool)
    split = np.flatnonzero(v.nodes["feature"] >= 0)
    v.nodes["value"][split[:8192]] = pool
    x = _rows(rng, N0 + 5, 1, pool, nan=0.05)
    _check(x, v, _trees(rng, 1, 8, 5, pool[:100]), 0.5, 64, launches=5)


@pytest.mark.parametrize("nan", [0.0, 0.2])
def test_half_tables(nan):
    rng = np.random.default_rng(9)
    pool = _pool(rng, 200)
    x = _rows(rng, N0 + 77, 6, pool, nan=nan)
    x[:50] *= 1e5  # past binary16's range
    _check(x, _trees(rng, 6, 20, 7, pool), _trees(rng, 6, 30, 7, pool, split=0.7), 0.5, 64, half=True)


def test_threshold_extremes():
    rng = np.random.default_rng(3)
    f32 = np.float32
    pool = np.array([0.0, -0.0, 1e-45, -1e-45, 3.4028235e38, -3.4028235e38, 1.17549435e-38, 1.0], dtype=f32)
    x = _rows(rng, N0 + 9, 4, pool, nan=0.1)
    _check(x, _trees(rng, 4, 20, 6, pool), _trees(rng, 4, 20, 6, pool), 0.5, 64)


def test_accumulation_batches():
    import torch

    rng = np.random.default_rng(21)
    pool = _pool(rng, 90)
    n, batch, F = 3 * N0 + 100, N0 + 40, 5
    x = _rows(rng, n, F, pool, nan=0.01)
    v, p = _trees(rng, F, 20, 6, pool), _trees(rng, F, 20, 6, pool)
    opv, opf, valid, _ = O.screen_rows(x, v, p, 0.5)
    mlt.set_num_features(F)
    mlt.load_ensemble(mlt.MLT_MODEL_V, v.nodes, v.n_trees, v.depth)
    mlt.load_ensemble(mlt.MLT_MODEL_P, p.nodes, p.n_trees, p.depth)
    target = int(valid[:batch].sum()) + 1  # reached in the second batch
    _, pf, tk, stats = mlt.screen_until(torch.from_numpy(x).cuda(), batch, target, 0.5, 50)
    mlt.sync_status()
    used = 2 * batch
    assert stats.cpu().tolist() == [used, int(valid[:used].sum()), 2]
    assert np.array_equal(pf.cpu().numpy()[:used].view(np.uint32), opf[:used].view(np.uint32))
    assert np.array_equal(tk.cpu().numpy(), O.topk(opf[:used], valid[:used], 50)[0])


@pytest.mark.parametrize("vd,pd,split", [(11, 14, 0.9), (12, 11, 0.97), (13, 13, 0.6), (14, 12, 0.8), (5, 14, 0.75)])
@pytest.mark.parametrize("nan", [0.0, 0.2])
def test_deep_models(vd, pd, split, nan):
    """Heads, exits and tail blocks: leaves at every level of a block, paths
    that end in the head, at an exit and at the bottom."""
    rng = np.random.default_rng(100 * vd + pd)
    F = 3 + vd % 4
    pool = _pool(rng, 400)
    x = _rows(rng, N0 + 47, F, pool, nan=nan)
    v = _trees(rng, F, 61, vd, pool, split=split if vd > 10 else 1.0)
    _check(x, v, _trees(rng, F, 70, pd, pool, split=split), 0.5, 100)


@pytest.mark.parametrize("trees", [1, 4, 7, 8, 9, 49, 100])
def test_deep_tree_counts(trees):
    rng = np.random.default_rng(trees)
    pool = _pool(rng, 60)
    x = _rows(rng, N0, 1, pool, nan=0.1)
    v = _trees(rng, 1, 20, 11, pool, split=0.9)
    p = _trees(rng, 1, trees, 12, pool, split=0.95)
    _check(x, v, p, 0.5, 64, launches=6)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 500, 4097])
@pytest.mark.parametrize("vd,pd", [(6, 6), (4, 10), (12, 13)])
def test_small_batches(n, vd, pd):
    """Tiles of one block, more tree groups than trees, waves with idle CTAs."""
    rng = np.random.default_rng(n + vd)
    pool = _pool(rng, 100)
    mlt.tune_fused_small(0)
    try:
        x = _rows(rng, n, 9, pool, nan=0.05, special=n > 40)
        v, p = (_trees(rng, 9, t, d, pool, split=0.95 if d > 10 else 1.0) for t, d in ((37, vd), (5, pd)))
        _check(x, v, p, 0.5, 64)
    finally:
        mlt.tune_fused_small(8192)


@pytest.mark.parametrize("F,n,trees,depth,launches", [
    (20, 13397, 500, 5, 6), (24, 3818, 107, 7, 4), (82, 43767, 56, 6, 4), (64, 65536, 200, 8, 6), (30, 200, 900, 8, 4)])
def test_rule(F, n, trees, depth, launches):
    """Which batches take the ordinal walk by default (two more launches)."""
    import torch

    mlt.tune_ordinal(1)
    rng = np.random.default_rng(1)
    e = _trees(rng, F, trees, depth, _pool(rng, 500))
    mlt.set_num_features(F)
    for m in (mlt.MLT_MODEL_V, mlt.MLT_MODEL_P):
        mlt.load_ensemble(m, e.nodes, e.n_trees, e.depth)
    before = mlt.kernel_launches()
    mlt.screen(torch.zeros((n, F), device="cuda"), 0.5, 10)
    mlt.sync_status()
    assert mlt.kernel_launches() - before == launches


def test_the_form_is_packed_beside_the_table():
    """Loading a V model costs little more than loading the same trees as model
    A, which has no ordinal form."""
    import time

    cfg = W.ScreenConfig(4, "load", 64, 96, 300, 10, 300, 10, 0.5, 16, None)
    e = W.make_ensemble(cfg, "V", W._RangeThresholds([(0.0, 1.0)] * 96), 3)
    mlt.set_num_features(96)
    best = {}
    for _ in range(7):
        for m in (mlt.MLT_MODEL_V, mlt.MLT_MODEL_A):
            t = time.perf_counter()
            mlt.load_ensemble(m, e.nodes, e.n_trees, e.depth)
            best[m] = min(best.get(m, 1e9), time.perf_counter() - t)
    mlt.free_ensemble(mlt.MLT_MODEL_A)
    assert best[mlt.MLT_MODEL_V] < 2.0 * best[mlt.MLT_MODEL_A], best


@pytest.mark.parametrize("F,n,v,p", [(20, 13397, (500, 5), (500, 5)), (64, 65536, (200, 8), (20, 4)),
                                     (47, 20011, (20, 5), (300, 14)), (30, 200, (900, 8), (900, 8))])
def test_shape_query_agrees_with_the_launches(F, n, v, p):
    """A pass has an ordinal shape exactly where it takes one more launch."""
    import torch

    mlt.tune_ordinal(1)
    rng = np.random.default_rng(2)
    mlt.set_num_features(F)
    for m, (trees, depth) in ((mlt.MLT_MODEL_V, v), (mlt.MLT_MODEL_P, p)):
        e = _trees(rng, F, trees, depth, _pool(rng, 500), split=0.75 if depth > 10 else 1.0)
        mlt.load_ensemble(m, e.nodes, e.n_trees, e.depth)
    mlt.tune_fused_small(0)
    try:
        before = mlt.kernel_launches()
        mlt.screen(torch.zeros((n, F), device="cuda"), 0.5, 10)
        mlt.sync_status()
        launches = mlt.kernel_launches() - before
    finally:
        mlt.tune_fused_small(8192)
    shapes = [mlt.ordinal_shape(mlt.MLT_MODEL_V, n), mlt.ordinal_shape(mlt.MLT_MODEL_P, n, True)]
    assert launches == 4 + sum(s is not None for s in shapes), shapes
    assert all(s is None or s["candidates"] * s["splits"] <= 1024 for s in shapes), shapes
    mlt.tune_ordinal(0)
    assert mlt.ordinal_shape(mlt.MLT_MODEL_P, n, True) is None


@pytest.mark.parametrize("n", [20001, 20033, 20127])
@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("nan", [0.0, 0.05])
def test_wide_items(n, half, nan):
    """Aligned batches large enough for 128 rows an item (the others here take
    64), ending inside one."""
    import torch

    F = 256
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n // 128 * (F // 8) >= sms * 32  # the rule of launch_ordinals
    rng = np.random.default_rng(n)
    pool = _pool(rng, 150)
    x = _rows(rng, n, F, pool, nan=nan)
    _check(x, _trees(rng, F, 60, 7, pool), _trees(rng, F, 60, 7, pool), 0.5, 64, half=half)


@pytest.mark.parametrize("F", [4, 12, 40])
def test_half_tables_of_aligned_rows(F):
    rng = np.random.default_rng(F)
    pool = _pool(rng, 200)
    x = _rows(rng, N0 + 61, F, pool, nan=0.05)
    _check(x, _trees(rng, F, 30, 7, pool), _trees(rng, F, 30, 7, pool), 0.5, 64, half=True)
