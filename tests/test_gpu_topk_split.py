"""The split top-k where it really splits (k <= 256: lists of more than 20,480
scores): batches of uneven lists, where some are cut into slices and merged
and others finished by one CTA of the same launch, against the oracle's sort;
one workspace shared by unsynchronised score -> slices -> merge passes; and a
long list among short ones spread over the GPU."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from tests import gpu_cases as gc

pytestmark = pytest.mark.gpu


def _lists(seed):
    """An empty list, one shorter than most k, both sides of the length that is
    not cut, long ones (ties, NaN, -inf), and sorted ones, whose top lies in one
    slice."""
    g = np.random.default_rng(seed)
    lists = []
    for n in (0, 7, 1000, 20_480, 20_481, 61_003, 150_000):
        x = np.round(g.standard_normal(n) * 50, 1).astype(np.float32)
        x[g.random(n) < 0.01] = -np.inf
        x[g.random(n) < 0.01] = np.nan
        lists.append(x)
    lists += [np.arange(70_000, dtype=np.float32), -np.arange(70_000, dtype=np.float32),
              np.full(50_000, 2.5, np.float32)]
    return lists


@pytest.mark.parametrize("k", [1, 10, 100, 128, 256])
def test_uneven_batches_match_the_oracle(cuda_lib, k):
    import torch
    from paper_2606_26439_gb300 import tms
    lists = _lists(k)
    want = {id(x): oracle.topk(x.astype(np.float64), k) for x in lists}
    for batch in (lists, lists[5:7], lists[6:7], [lists[2]] * 9 + [lists[6]] * 3):
        co = np.zeros(len(batch) + 1, np.int64)
        co[1:] = np.cumsum([len(x) for x in batch])
        n = int(co[-1])
        s, off = gc.to_dev(np.concatenate(batch), co)
        need = tms.topk_workspace_size(len(batch), k, n)
        assert need > 0
        ws = torch.full((need,), 0x5A, dtype=torch.uint8, device="cuda")  # stale contents must not matter
        got = [tms.topk_split(s, off, k, n_cand=n, workspace=ws), tms.topk_split_noalloc(s, off, k, n_cand=n)]
        torch.cuda.synchronize()
        assert tms.device_error() == 0
        for i, x in enumerate(batch):
            want_s, want_p = want[id(x)]
            for ts, tp in got:
                assert np.array_equal(tp[i].cpu().numpy(), want_p), i
                v = ts[i].cpu().numpy().astype(np.float64)
                assert ((v == want_s) | (np.isnan(v) & np.isnan(want_s))).all(), i


def test_chained_slices_and_merges_share_one_workspace(cuda_lib):
    """Score -> slices -> merge passes with nothing between them, over one score
    buffer and one workspace: every pass as if run alone."""
    import torch
    from paper_2606_26439_gb300 import tms
    dev, n_docs, n, k, passes = torch.device("cuda"), 40_000, 30_000, 16, 12
    tok, off, ln = synth.device_dense_corpus(synth.lengths_uniform(n_docs, 1, 24, 72), 64, "f16", 72, dev)
    qs = [synth.queries(2, 32, 64, "f16", 400 + i).to(dev) for i in range(passes)]
    lists = [torch.from_numpy(np.concatenate([synth.candidates(n_docs, n, 500 + i, j) for j in range(2)])
                              .astype(np.int32)).to(dev) for i in range(passes)]
    co = torch.tensor([0, 1000, 2 * n], dtype=torch.int64, device=dev)  # one list cut, one not
    need = tms.topk_workspace_size(2, k, 2 * n)
    assert need > 0
    ws = torch.empty(need, dtype=torch.uint8, device=dev)
    out = torch.empty(2 * n, dtype=torch.float32, device=dev)
    ts = torch.empty((passes, 2, k), dtype=torch.float32, device=dev)
    tp = torch.empty((passes, 2, k), dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    for i in range(passes):
        tms.score_dense(qs[i], tok, off, ln, lists[i], co, out=out)
        tms.topk_split(out, co, k, 2 * n, ts[i], tp[i], ws)
    torch.cuda.synchronize()
    assert tms.device_error() == 0
    for i in range(passes):
        alone = tms.score_dense(qs[i], tok, off, ln, lists[i], co)
        torch.cuda.synchronize()
        want_s, want_p = tms.topk(alone, co, k)
        torch.cuda.synchronize()
        assert torch.equal(tp[i], want_p) and torch.equal(ts[i].view(torch.int32), want_s.view(torch.int32)), i


def test_a_long_list_among_short_ones_is_cut(cuda_lib):
    """31 lists of 600 scores and one of 600,000: 0.15 of the time that one CTA
    for each list takes (1.0 when the slices went by the average length)."""
    import torch
    from paper_2606_26439_gb300 import tms
    co = np.concatenate([[0], np.cumsum([600_000] + [600] * 31)])
    n = int(co[-1])
    s, off = gc.to_dev(np.random.default_rng(1).standard_normal(n).astype(np.float32), co.astype(np.int64))
    ws = torch.empty(max(16, tms.topk_workspace_size(32, 10, n)), dtype=torch.uint8, device="cuda")
    t = []
    for f in (lambda: tms.topk(s, off, 10), lambda: tms.topk_split(s, off, 10, n, workspace=ws)):
        best = float("inf")
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                f()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        t.append(best)
    assert t[1] < 0.5 * t[0], t
