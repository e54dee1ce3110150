"""Rerank on both sides of the size at which the last walk CTA stops ordering
the keys itself (512), with duplicates, empty slots, more wanted than there
are, repeated calls, arrivals left over from a call that stopped part-way, and
replays of a captured call."""
import numpy as np
import pytest

import oracle as O
from paper_2411_10764_gb300 import mlt
from paper_2411_10764_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 31, 33, 128, 511, 512, 513, 2000])
@pytest.mark.parametrize("trees,depth", [(40, 5), (300, 14)])
def test_sizes(m, trees, depth):
    import torch

    w = W.make_workload(1, seed=5, n=3000)
    a = W.make_model_a(w, seed=5, n_trees=trees, depth=depth)
    rng = np.random.default_rng(m)
    mlt.set_num_features(w.feats.shape[1])
    mlt.load_ensemble(mlt.MLT_MODEL_A, a.nodes, a.n_trees, a.depth)
    x = torch.from_numpy(w.feats).cuda()
    for call in range(3):
        cand = rng.integers(0, w.n, m).astype(np.int64)
        cand[rng.random(m) < 0.1] = -1
        n_final = max(1, [m // 2, m, m + 9][call])
        score, final = mlt.rerank(x, torch.from_numpy(cand).cuda(), n_final)
        mlt.sync_status()
        es, ef = O.rerank(w.feats, cand, a, n_final)
        assert np.array_equal(score.cpu().numpy().view(np.uint32), es.view(np.uint32))
        assert np.array_equal(final.cpu().numpy(), ef)


@pytest.mark.parametrize("left", [1, 127, 128, 0xFFFF])
def test_left_over_arrivals_do_not_reach_the_next_call(left):
    import torch

    w = W.make_workload(1, seed=6, n=3000)
    a = W.make_model_a(w, seed=6, n_trees=40, depth=5)
    rng = np.random.default_rng(left)
    mlt.set_num_features(w.feats.shape[1])
    mlt.load_ensemble(mlt.MLT_MODEL_A, a.nodes, a.n_trees, a.depth)
    x = torch.from_numpy(w.feats).cuda()
    for _ in range(2):
        cand = rng.integers(0, w.n, 128).astype(np.int64)
        final = torch.full((64,), -7, dtype=torch.int64, device="cuda")
        mlt.selftest_poison_state(left)
        score, final = mlt.rerank(x, torch.from_numpy(cand).cuda(), 64, out_final=final)
        mlt.sync_status()
        es, ef = O.rerank(w.feats, cand, a, 64)
        assert np.array_equal(score.cpu().numpy().view(np.uint32), es.view(np.uint32))
        assert np.array_equal(final.cpu().numpy(), ef)


def test_replays_of_a_captured_call():
    import torch

    w = W.make_workload(1, seed=7, n=3000)
    a = W.make_model_a(w, seed=7, n_trees=40, depth=5)
    mlt.set_num_features(w.feats.shape[1])
    mlt.load_ensemble(mlt.MLT_MODEL_A, a.nodes, a.n_trees, a.depth)
    x = torch.from_numpy(w.feats).cuda()
    cand = torch.zeros(128, dtype=torch.int64, device="cuda")
    score, final = mlt.rerank(x, cand, 64)
    mlt.sync_status()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        mlt.rerank(x, cand, 64, out_score=score, out_final=final)
    rng = np.random.default_rng(7)
    for _ in range(3):
        c = rng.integers(0, w.n, 128).astype(np.int64)
        cand.copy_(torch.from_numpy(c))
        final.fill_(-7)
        g.replay()
        mlt.sync_status()
        es, ef = O.rerank(w.feats, c, a, 64)
        assert np.array_equal(score.cpu().numpy().view(np.uint32), es.view(np.uint32))
        assert np.array_equal(final.cpu().numpy(), ef)
