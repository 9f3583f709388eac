"""Long queries, where the query tile and the row maxima compete with the
chunk stages for shared memory: scores against the oracle and bit for bit
against one call for each list, and times against a neighbouring shape, which
show a launch with too few stages."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from tests import gpu_cases as gc
from tests.test_gpu_dealing import best_time

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,nq,d", [("f16", 128, 448), ("bf16", 96, 640), ("f16", 64, 960), ("f16", 100, 704),
                                        ("fp8", 128, 896), ("fp8", 97, 128), ("fp8", 128, 64), ("fp8", 128, 144)])
def test_long_queries(cuda_lib, dtype, nq, d):
    import torch
    from paper_2606_26439_gb300 import tms
    base = "f16" if dtype == "fp8" else dtype
    tok, off, ln = gc.edge_corpus(d, base, 600 + d)
    cands = [np.random.default_rng(d + i).permutation(len(ln))[:n].astype(np.int32)
             for i, n in enumerate((len(ln), 0, 3, 40, 1))]
    Q = synth.queries(len(cands), nq, d, base, 601 + d)
    flat, co = gc.csr(cands)
    q, t, o, l, f, c = gc.to_dev(Q, tok, off, ln, flat, co)
    if dtype == "fp8":
        (qc, qs), (tc, ts) = tms.quantize_e4m3(q), tms.quantize_e4m3(t)
        q, t = (qc, qs), (tc, ts)
        score = lambda i, ids, offs: tms.score_fp8(qc[i], qs[i], tc, ts, o, l, ids, offs)  # noqa: E731
        dq = qc.cpu().view(torch.float8_e4m3fn).float() * qs.cpu().unsqueeze(-1)
        dt = tc.cpu().view(torch.float8_e4m3fn).float() * ts.cpu().unsqueeze(-1)
    else:
        score = lambda i, ids, offs: tms.score_dense(q[i], t, o, l, ids, offs)  # noqa: E731
        dq, dt = Q, tok
    got = score(slice(None), f, c).cpu().numpy()
    for i, x in enumerate(cands):
        if len(x):
            ids, offs = gc.to_dev(x, np.array([0, len(x)], np.int64))
            one = score(slice(i, i + 1), ids, offs).cpu().numpy()
            assert np.array_equal(got[co[i]:co[i + 1]].view(np.uint32), one.view(np.uint32))
    assert tms.device_error() == 0
    want = gc.oracle_dense_multi(dq, dt, off, ln, cands)
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    fin = np.isfinite(want)
    assert (np.abs(got[fin] - want[fin]) <= 1e-3 * np.maximum(np.abs(want[fin]), nq * 1e-3)).all()


def _lists(n, cand, docs):
    import torch
    ids = torch.cat([synth.device_candidates(docs, cand, 83, i) for i in range(n)]).to(torch.int32)
    return ids, torch.arange(n + 1, dtype=torch.int64, device="cuda") * cand


def test_a_resident_query_leaves_stages_for_the_documents(cuda_lib):
    """128 query tokens, d = 448 against d = 384: 1.2 times for 1.17 times the
    bytes (1.4 with the two stages that the resident tile leaves)."""
    import torch
    from paper_2606_26439_gb300 import tms
    t = []
    for d in (384, 448):
        tok, off, ln = synth.device_dense_corpus(synth.lengths_uniform(20_000, 32, 180, 83), d, "f16", 83)
        q = synth.device_unit_rows(4 * 128, d, "f16", 83, 1).view(4, 128, d)
        ids, co = _lists(4, 8000, 20_000)
        out = torch.empty(len(ids), device="cuda")
        t.append(best_time(lambda: tms.score_dense(q, tok, off, ln, ids, co, out=out)))
    assert t[1] < 1.3 * t[0], t


def test_four_query_blocks_on_short_documents(cuda_lib):
    """80,000 FP8 documents of 16 tokens against 128 query tokens: 156 us (281
    when one warp summed a document's four query blocks one after the other,
    251 when four warps did)."""
    import torch
    from paper_2606_26439_gb300 import tms
    tok, off, ln = synth.device_dense_corpus(synth.lengths_fixed(20_000, 16), 128, "f16", 84)
    tc, ts = tms.quantize_e4m3(tok)
    qc, qs = tms.quantize_e4m3(synth.device_unit_rows(8 * 128, 128, "f16", 84, 1).view(8, 128, 128))
    ids, co = _lists(8, 10_000, 20_000)
    out = torch.empty(len(ids), device="cuda")
    assert best_time(lambda: tms.score_fp8(qc, qs, tc, ts, off, ln, ids, co, out=out)) < 220
