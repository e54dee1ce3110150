"""Batched accumulation screens groups of batches at once: the batch that
reaches the target must still be the last one consumed, wherever in a group it
lies, and nothing past it written; and where a batch alone keeps the GPU busy,
no group holds a second one for V to walk in vain."""
import numpy as np
import pytest

import oracle as O
from paper_2411_10764_gb300 import mlt
from paper_2411_10764_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 80000  # two groups of small batches


@pytest.fixture(scope="module")
def problem():
    w = W.make_workload(1, seed=11, n=N)
    pv, pf, valid, _ = O.screen_rows(w.feats, w.v, w.p, w.thr)
    return w, pv, pf, valid


def _run(w, batch, target, k, with_outputs=True):
    import ctypes as C

    import torch

    mlt.load_workload_models(w)
    x = torch.from_numpy(w.feats).cuda()
    pv = torch.full((w.n,), -7.0, device="cuda") if with_outputs else None
    pf = torch.full((w.n,), -7.0, device="cuda") if with_outputs else None
    tk = torch.empty(k, dtype=torch.int64, device="cuda")
    st = torch.empty(3, dtype=torch.int64, device="cuda")
    ptr = lambda t: C.c_void_p(0 if t is None else t.data_ptr())
    rc = mlt.lib().mlt_screen_until(C.c_void_p(torch.cuda.current_stream().cuda_stream), ptr(x), w.n, batch, target,
                                    C.c_float(w.thr), k, ptr(pv), ptr(pf), ptr(tk), ptr(st))
    assert rc == 0
    mlt.sync_status()
    return pv, pf, tk.cpu().numpy(), st.cpu().tolist()


@pytest.mark.parametrize("batch", [7, 500, 1000, 8192, 24576, 24577, 30000, 80000, 100000])
@pytest.mark.parametrize("where", ["first", "exact", "past", "middle", "late", "never"])
def test_cut(problem, batch, where):
    w, opv, opf, valid = problem
    total = np.cumsum(valid)
    first = int(total[min(batch, N) - 1])
    target = {"first": 1, "exact": max(1, first), "past": first + 1, "middle": int(total[-1] * 0.4),
              "late": int(total[-1]), "never": int(total[-1]) + 1}[where]
    ends = np.append(np.arange(batch, N, batch), N)
    counts = total[ends - 1]
    j = min(int(np.searchsorted(counts, target)), len(ends) - 1)
    used = int(ends[j])
    if -(-N // batch) > 65536:
        pytest.skip("more batches than a call takes")
    pv, pf, tk, stats = _run(w, batch, target, 100)
    assert stats == [used, int(counts[j]), j + 1]
    pv, pf = pv.cpu().numpy(), pf.cpu().numpy()
    assert np.array_equal(pf[:used].view(np.uint32), opf[:used].view(np.uint32))
    assert np.all(np.abs(pv[:used].astype(np.float64) - opv[:used]) <= 1e-6 * np.maximum(np.abs(opv[:used]), 1e-30))
    assert np.all(pv[used:] == -7.0) and np.all(pf[used:] == -7.0)
    assert np.array_equal(tk, O.topk(opf[:used], valid[:used], 100)[0])
    assert mlt.last_survivor_count() == int(counts[j]) - (int(counts[j - 1]) if j else 0)


def test_no_outputs(problem):
    w, _, opf, valid = problem
    target = int(valid[:30000].sum())
    _, _, tk, stats = _run(w, 1000, target, 64, with_outputs=False)
    assert stats[0] <= 30000 and stats[1] >= target
    assert np.array_equal(tk, O.topk(opf[:stats[0]], valid[:stats[0]], 64)[0])


def _launches(n, batch):
    """Kernels of one accumulation call over the loaded models (zero rows)."""
    import torch

    x = torch.zeros((n, 64), device="cuda")
    mlt.screen_until(x, batch, 1 << 30, 0.5, 16, with_outputs=False)  # buffers and plans
    before = mlt.kernel_launches()
    mlt.screen_until(x, batch, 1 << 30, 0.5, 16, with_outputs=False)
    mlt.sync_status()
    return mlt.kernel_launches() - before


def _load(vt, vd, pt, pd):
    mlt.set_num_features(64)
    for m, trees, depth in ((mlt.MLT_MODEL_V, vt, vd), (mlt.MLT_MODEL_P, pt, pd)):
        e = W.make_ensemble(W.ScreenConfig(2, "groups", 64, 64, vt, vd, pt, pd, 0.5, 16, 0.5), "V" if m == mlt.MLT_MODEL_V
                            else "P", W._RangeThresholds([(0.0, 1.0)] * 64), 7, n_trees=trees, depth=depth)
        mlt.load_ensemble(m, e.nodes, e.n_trees, e.depth)


@pytest.mark.parametrize("vt,vd,pt,pd,batch,batches,groups,cuts", [
    (1000, 12, 300, 12, 24576, 4, 4, 0),  # a batch fills the GPU: one a group
    (1000, 8, 100, 6, 32768, 3, 3, 0),
    (1000, 12, 300, 12, 8192, 3, 2, 1),   # two batches, then the third
    (1000, 12, 300, 12, 8192, 5, 2, 2),   # two batches, then three
    (50, 6, 100, 6, 24576, 2, 1, 1),      # cheap walks: both together
    (50, 6, 100, 6, 500, 40, 1, 1),
])
def test_groups(vt, vd, pt, pd, batch, batches, groups, cuts):
    """`cuts` groups hold several batches and take a cut each."""
    _load(vt, vd, pt, pd)
    mlt.tune_ordinal(0)  # one launch a walk whatever the group's size
    try:
        one = _launches(batch, batch)
        # two batches as large as these are two groups whatever the models
        per = _launches(1 << 21, 1 << 20) - _launches(1 << 20, 1 << 20)
        assert _launches(batches * batch, batch) - one == (groups - 1) * per + cuts
    finally:
        mlt.tune_ordinal(1)


@pytest.mark.parametrize("vt,vd,batch", [(400, 12, 24583), (400, 12, 4000), (1500, 8, 24576)])
@pytest.mark.parametrize("hit", [1, 2, 4])
def test_deep_models_equal_screening_of_the_prefix(vt, vd, batch, hit):
    """Groups of one batch and of several, V and P in ordinal form."""
    import torch

    _load(vt, vd, 60, 12)
    n = 4 * batch + 11
    x = torch.rand((n, 64), device="cuda", generator=torch.Generator(device="cuda").manual_seed(batch))
    _, pf, _ = mlt.screen(x, 0.5, 16)
    counts = torch.cumsum(torch.isfinite(pf).long(), 0)
    target = int(counts[hit * batch - 1]) if hit > 1 else 1
    used = int((counts >= target).nonzero()[0]) // batch * batch + batch
    pv, pf, tk, stats = mlt.screen_until(x, batch, target, 0.5, 100)
    wv, wf, wk = mlt.screen(x[:used].contiguous(), 0.5, 100)
    mlt.sync_status()
    assert stats.cpu().tolist() == [used, int(counts[used - 1]), used // batch]
    assert torch.equal(pv[:used], wv) and torch.equal(pf[:used], wf) and torch.equal(tk, wk)
