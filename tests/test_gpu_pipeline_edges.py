"""Where the scoring pipeline's packing and dealing change form, on the GPU:
documents around the 8-row units and the 128 / 256-row super-tiles, queries
that change with every super-tile, query groups dealt to the CTAs in one or
several rounds, and fp32 shapes on both sides of the tensor-memory query and
of the exact kernel.  All comparisons are bit for bit: a call over many lists
against one call for each, and shared lists against per-query lists (parity
with the FP64 oracle over shapes and types is test_gpu_dense's)."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from tests import gpu_cases as gc

pytestmark = pytest.mark.gpu

LENGTHS = [1, 7, 8, 9, 15, 16, 17, 120, 121, 127, 128, 129, 136, 248, 255, 256, 257, 384, 1000]


def _corpus(d, dtype, seed):
    ln = np.array((LENGTHS + [8] * 40 + [3] * 40 + [256, 128, 128]) * 2, np.int32)
    return synth.dense_corpus(len(ln), ln, d, dtype, seed)


@pytest.mark.parametrize("dtype,nq,d", [("f16", 32, 128), ("bf16", 17, 64), ("f16", 70, 128), ("f16", 128, 256),
                                        ("f32", 32, 128), ("f32", 1, 8), ("f32", 96, 96), ("f32", 128, 128),
                                        ("f32", 32, 136), ("f32", 32, 544), ("f32", 32, 552), ("f32", 96, 200)])
def test_units_and_query_changes(cuda_lib, dtype, nq, d):
    """Lists of one to three documents per query (a query change at every
    super-tile), then one list of everything in random order: the same bits
    as one call for each list, where no query follows another."""
    tok, off, ln = _corpus(d, dtype, 900 + nq + d)
    g = np.random.default_rng(nq + d)
    cands = [g.integers(0, len(ln), n).astype(np.int32) for n in g.integers(0, 4, 40)]
    cands.append(g.permutation(len(ln)).astype(np.int32))
    Q = synth.queries(len(cands), nq, d, dtype, 900 + d)
    got, flags = gc.gpu_dense(Q, tok, off, ln, cands)
    assert flags == 0
    single = []
    for i, c in enumerate(cands):
        if len(c):
            one, flags = gc.gpu_dense(Q[i:i + 1], tok, off, ln, [c])
            assert flags == 0
            single.append(np.asarray(one, np.float32))
    got = np.asarray(got, np.float32)
    assert np.isfinite(got).all()
    assert np.array_equal(got.view(np.uint32), np.concatenate(single).view(np.uint32))


@pytest.mark.parametrize("n_queries", [2, 5, 8, 9, 17, 40, 57, 130, 300])
@pytest.mark.parametrize("n_cand", [1, 3, 400])
def test_shared_rounds_equal_per_query_lists(cuda_lib, n_queries, n_cand):
    """Any number of groups and candidates, empty and bad documents among
    them: the same bits as per-query lists, fp16 and FP8."""
    import torch
    from paper_2606_26439_gb300 import tms
    tok, off, ln = _corpus(128, "f16", 77)
    ln = ln.copy()
    ln[5] = 0
    g = np.random.default_rng(n_queries + n_cand)
    cand = g.integers(0, len(ln), n_cand).astype(np.int32)
    if n_cand > 3:
        cand[:2] = (5, len(ln))  # empty, bad id
    Q = synth.queries(n_queries, 29, 128, "f16", 78)
    q, t, o, l, c, cc, co = gc.to_dev(Q, tok, off, ln, cand, np.tile(cand, n_queries),
                                      np.arange(n_queries + 1, dtype=np.int64) * n_cand)
    shared = tms.score_dense_shared(q, t, o, l, c)
    lists = tms.score_dense(q, t, o, l, cc, co).view(n_queries, n_cand)
    assert torch.equal(shared.view(torch.int32), lists.view(torch.int32))
    qc, qs = tms.quantize_e4m3(q)
    tc, ts = tms.quantize_e4m3(t)
    shared = tms.score_fp8_shared(qc, qs, tc, ts, o, l, c)
    lists = tms.score_fp8(qc, qs, tc, ts, o, l, cc, co).view(n_queries, n_cand)
    assert torch.equal(shared.view(torch.int32), lists.view(torch.int32))
    assert tms.device_error() & ~tms.TMS_DEVERR_BAD_ID == 0


@pytest.mark.parametrize("n_queries", [2, 4, 7])
@pytest.mark.parametrize("d", [64, 96, 192, 256, 320, 640])
def test_shared_row_lengths_equal_per_query_lists(cuda_lib, n_queries, d):
    """Both sides of each row length at which the super-tile, the CTAs per SM
    or the query tile (resident, streamed) changes: the same bits as
    per-query lists, fp16 and FP8."""
    import torch
    from paper_2606_26439_gb300 import tms
    tok, off, ln = _corpus(d, "f16", 500 + d)
    cand = np.random.default_rng(d).permutation(len(ln)).astype(np.int32)
    Q = synth.queries(n_queries, 32, d, "f16", 501 + d)
    q, t, o, l, c, cc, co = gc.to_dev(Q, tok, off, ln, cand, np.tile(cand, n_queries),
                                      np.arange(n_queries + 1, dtype=np.int64) * len(cand))
    shared = tms.score_dense_shared(q, t, o, l, c)
    lists = tms.score_dense(q, t, o, l, cc, co).view(n_queries, -1)
    assert torch.equal(shared.view(torch.int32), lists.view(torch.int32))
    qc, qs = tms.quantize_e4m3(q)
    tc, ts = tms.quantize_e4m3(t)
    shared = tms.score_fp8_shared(qc, qs, tc, ts, o, l, c)
    lists = tms.score_fp8(qc, qs, tc, ts, o, l, cc, co).view(n_queries, -1)
    assert torch.equal(shared.view(torch.int32), lists.view(torch.int32))
    assert tms.device_error() == 0


@pytest.mark.parametrize("M,K", [(16, 256), (16, 255), (16, 252), (16, 3), (32, 128), (32, 126), (32, 20)])
@pytest.mark.parametrize("lists", [(1,), (0, 1, 0, 2), (700, 1, 0, 3, 150, 151, 152, 153), (5, 1500), (1,) * 200],
                         ids=["one", "few", "uneven", "two", "many"])
@pytest.mark.parametrize("f16", [False, True])
def test_pq_shares_and_table_rows_exact(cuda_lib, M, K, lists, f16):
    """Lists of every size cut over the CTAs, tables whose rows are and are
    not 16-byte aligned: an integer-valued table (exact in fp16 and in every
    partial sum) must give the exact scores, every candidate written once."""
    import torch
    from paper_2606_26439_gb300 import tms
    g = np.random.default_rng(M + K + len(lists))
    nq, nd = 19, 60
    T = g.integers(-1000, 1001, size=(len(lists), nq, M, K)).astype(np.float32)
    ln = g.integers(0, 40, nd).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(ln)[:-1]]).astype(np.int64)
    codes = g.integers(0, K, size=(int(ln.sum()), M)).astype(np.uint8)
    cands = [g.integers(0, nd, n).astype(np.int32) for n in lists]
    flat, co = gc.csr(cands)
    t_d, c_d, o_d, l_d, f_d, co_d = gc.to_dev(T, codes, off, ln, flat, co)
    out = torch.full((len(flat),), 12345.5, dtype=torch.float32, device="cuda")
    tms.score_pq(t_d, c_d, o_d, l_d, f_d, co_d, out=out, f16_table=f16)
    got = out.cpu().numpy()
    assert tms.device_error() == 0
    for q, c in enumerate(cands):
        per_doc = np.full(nd, -np.inf)
        for x in set(c.tolist()):
            if ln[x]:
                rows = codes[off[x]:off[x] + ln[x]].astype(int)
                dots = T[q][:, np.arange(M), rows].sum(-1)  # (nq, tokens)
                per_doc[x] = dots.max(1).sum()
        assert np.array_equal(got[co[q]:co[q + 1]], per_doc[c].astype(np.float32))


@pytest.mark.parametrize("dtype", ["f16", "f32", "fp8"])
@pytest.mark.parametrize("lists", [(0, 0, 5), (1,) * 70, (0, 1, 0, 2, 0), (400, 1, 0, 3, 150, 151, 152, 153, 304),
                                   (2,) * 1100, (1, 3000, 1)], ids=["last", "ones", "few", "uneven", "many", "long"])
def test_lists_cut_over_ctas(cuda_lib, dtype, lists):
    """Lists of every size, empty ones between, cut over the CTAs: each
    candidate is written once, with the bits that its query and document give
    in a list of all documents."""
    import torch
    from paper_2606_26439_gb300 import tms
    tok, off, ln = _corpus(64, "f32" if dtype == "f32" else "f16", 88)
    g = np.random.default_rng(len(lists))
    Q = synth.queries(len(lists), 9, 64, "f32" if dtype == "f32" else "f16", 89)
    cands = [g.integers(0, len(ln), n).astype(np.int32) for n in lists]
    flat, co = gc.csr(cands)
    every = np.arange(len(ln), dtype=np.int32)
    q, t, o, l, f, c, e = gc.to_dev(Q, tok, off, ln, flat, co, every)
    out = torch.full((len(flat),), 12345.0, dtype=torch.float32, device="cuda")
    if dtype == "fp8":
        qc, qs = tms.quantize_e4m3(q)
        tc, ts = tms.quantize_e4m3(t)
        tms.score_fp8(qc, qs, tc, ts, o, l, f, c, out=out)
        full = tms.score_fp8_shared(qc, qs, tc, ts, o, l, e)
    else:
        tms.score_dense(q, t, o, l, f, c, out=out)
        if dtype == "f32":  # no shared lists: one call for each query
            whole = torch.tensor([0, len(ln)], dtype=torch.int64, device="cuda")
            full = torch.stack([tms.score_dense(q[i:i + 1], t, o, l, e, whole) for i in range(len(lists))])
        else:
            full = tms.score_dense_shared(q, t, o, l, e)
    got, full = out.cpu().numpy(), full.cpu().numpy()
    assert tms.device_error() == 0
    want = np.concatenate([full[i][x] for i, x in enumerate(cands)])
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
