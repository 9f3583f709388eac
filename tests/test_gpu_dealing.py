"""How work is dealt to the CTAs where candidates are few or lists unlike one
another: results bit for bit against one call for each query, and times
against calls of the same work in a form that is easy to deal."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def best_time(f, n=20):
    """Shortest mean time of n back-to-back calls, in microseconds."""
    import torch
    f()
    best = float("inf")
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1000 / n)
    return best


@pytest.mark.parametrize("queries,cand", [(4096, 1), (600, 2), (256, 4), (67, 9), (150, 19)])
def test_shared_lists_of_few_candidates(cuda_lib, queries, cand):
    """Many groups of queries over a handful of documents: the scores of
    per-query lists, whatever the rounds."""
    import torch
    from paper_2606_26439_gb300 import tms
    tok, off, ln = synth.device_dense_corpus(synth.lengths_uniform(cand, 1, 180, 81), 128, "f16", 81)
    q = synth.device_unit_rows(queries * 32, 128, "f16", 81, 1).view(queries, 32, 128)
    ids = torch.arange(cand, dtype=torch.int32, device="cuda")
    got = tms.score_dense_shared(q, tok, off, ln, ids)
    want = tms.score_dense(q, tok, off, ln, ids.repeat(queries),
                           torch.arange(queries + 1, dtype=torch.int64, device="cuda") * cand)
    torch.cuda.synchronize()
    assert tms.device_error() == 0
    assert torch.equal(got.view(torch.int32).flatten(), want.view(torch.int32))


def test_one_shared_candidate_uses_every_cta(cuda_lib):
    """4,096 queries x 1 document against 256 x 16, the same work: 1.4 times
    (6 when a round took 16 groups of queries on as many CTAs)."""
    import torch
    from paper_2606_26439_gb300 import tms
    tok, off, ln = synth.device_dense_corpus(synth.lengths_fixed(16, 128), 128, "f16", 82)
    q = synth.device_unit_rows(4096 * 32, 128, "f16", 82, 1).view(4096, 32, 128)
    ids = torch.arange(16, dtype=torch.int32, device="cuda")
    out = torch.empty((4096, 1), device="cuda")
    one = best_time(lambda: tms.score_dense_shared(q, tok, off, ln, ids[:1], out=out))
    few = best_time(lambda: tms.score_dense_shared(q[:256], tok, off, ln, ids, out=out.view(256, 16)))
    assert one < 3 * few, (one, few)
