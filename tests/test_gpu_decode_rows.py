"""Decoded rows written by k_decode_rows at the edges of its tiles, and decoded batches screened from those rows,
bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2411_10764_gb300 import mlt
from paper_2411_10764_gb300 import workloads as W
from screening import assert_parity, assert_same_bits

pytestmark = pytest.mark.gpu


def _space(rng, knobs, F):
    radices = rng.integers(1, 6, knobs).astype(np.int32)
    radices[0] = 16
    opts = rng.integers(1, 64, int(radices.sum())).astype(np.float32)
    prog = np.zeros(F, dtype=W.OP_DTYPE)
    for f in range(F):
        a, b = (int(v) for v in rng.integers(-1, knobs + f, 2))
        prog[f] = (int(rng.integers(0, 12)), a, b, float(rng.integers(1, 9)))
    return radices, opts, prog


@pytest.mark.parametrize("F,knobs", [(1, 1), (3, 8), (4, 8), (30, 3), (96, 8), (101, 12), (200, 16), (256, 16)])
def test_rows_and_digits(F, knobs):
    rng = np.random.default_rng(F)
    radices, opts, prog = _space(rng, knobs, F)
    space = int(np.prod(radices.astype(np.int64)))
    for n in (1, 31, 33, 127, 129, 255, 257, 513, 40001):
        n = min(n, space)
        first = int(rng.integers(0, space - n + 1))
        knob, feat = mlt.decode_knobs(radices, opts, prog, first, n)
        mlt.sync_status()
        ok, of = O.features(radices, opts, prog, first, n)
        assert np.array_equal(knob.cpu().numpy(), ok)
        assert_same_bits(feat.cpu().numpy(), of, "features", nan_equal=True)


@pytest.mark.parametrize("n,first", [(1, 7), (3000, 123456), (8193, 40), (16384, 5), (30001, 999999)])
def test_screening_from_rows(n, first):
    """One launch (n <= 8,192) and the ordinal walk; top-k holds candidate
    indices."""
    import torch

    d = W.conv2d_decoder(3, 70)
    cfg = W.ScreenConfig(4, "rows", n, 70, 40, 6, 60, 6, 0.5, 200, None, decoded=True)
    th = W._RangeThresholds(d.ranges)
    v = W.make_ensemble(cfg, "V", th, 3, n_trees=40 if n <= 8192 else 200, depth=6)
    p = W.make_ensemble(cfg, "P", th, 3, n_trees=60 if n <= 8192 else 190, depth=6)
    mlt.set_num_features(70)
    mlt.load_ensemble(mlt.MLT_MODEL_V, v.nodes, v.n_trees, v.depth)
    mlt.load_ensemble(mlt.MLT_MODEL_P, p.nodes, p.n_trees, p.depth)
    pv, pf, tk = mlt.screen_decoded(d.radices, d.option_values, d.program, first, n, 0.5, 200)
    mlt.sync_status()
    got = pv.cpu().numpy(), pf.cpu().numpy(), tk.cpu().numpy(), mlt.last_survivor_count()
    _, x = O.features(d.radices, d.option_values, d.program, first, n)
    opv, opf, valid, _ = O.screen_rows(x, v, p, 0.5)
    otk, s = O.topk(opf, valid, 200, index_base=first)
    assert_parity(got, (opv, opf, otk, s))
    # a capture finds the buffers too small: the call decodes inside the walks
    # instead of allocating, and the replay gives the same results
    if n == 30001:
        mlt.free_ensemble(mlt.MLT_MODEL_A)
        mlt.set_num_features(71)
        mlt.set_num_features(70)  # gives the row and ordinal buffers back
        mlt.load_ensemble(mlt.MLT_MODEL_V, v.nodes, v.n_trees, v.depth)
        mlt.load_ensemble(mlt.MLT_MODEL_P, p.nodes, p.n_trees, p.depth)
        outs = [torch.zeros_like(t) for t in (pv, pf, tk)]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            mlt.screen_decoded(d.radices, d.option_values, d.program, first, n, 0.5, 200, out_pvalid=outs[0],
                               out_perf=outs[1], out_topk=outs[2])
        g.replay()
        mlt.sync_status()
        assert_parity((outs[0].cpu().numpy(), outs[1].cpu().numpy(), outs[2].cpu().numpy(), s), (opv, opf, otk, s))
        # with the buffers in place the capture holds the row decoder and the
        # ordinal walk; other calls in between leave the replay its results
        mlt.screen_decoded(d.radices, d.option_values, d.program, first, n, 0.5, 200)
        g2 = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g2):
            mlt.screen_decoded(d.radices, d.option_values, d.program, first, n, 0.5, 200, out_pvalid=outs[0],
                               out_perf=outs[1], out_topk=outs[2])
        mlt.screen(torch.zeros((n, 70), device="cuda"), 0.5, 200)
        for t in outs:
            t.zero_()
        g2.replay()
        mlt.sync_status()
        assert_parity((outs[0].cpu().numpy(), outs[1].cpu().numpy(), outs[2].cpu().numpy(), s), (opv, opf, otk, s))
