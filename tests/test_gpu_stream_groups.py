"""Batched accumulation screens groups of batches at once (24,576 candidates,
then twice as many each): the batch that reaches the target must still be the
last one consumed, wherever in a group it lies, and nothing past it written."""
import numpy as np
import pytest

import oracle as O
from paper_2411_10764_gb300 import mlt
from paper_2411_10764_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 80000  # groups of 24,576, 49,152 and the rest, in whole batches


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
