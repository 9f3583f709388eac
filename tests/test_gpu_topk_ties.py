"""Top-k where very many keys reach the bound that the selection takes from
the threads' largest keys: equal scores across the cut (with few, or none,
above them), and a bound that k or more keys exceed.  Bit-exact against the
oracle's sort; and a list of equal scores costs about what any list does."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from tests import gpu_cases as gc

pytestmark = pytest.mark.gpu


def _check(x, k):
    import torch
    from paper_2606_26439_gb300 import tms
    x = np.asarray(x, np.float32)
    s, co = gc.to_dev(x, np.array([0, len(x)], np.int64))
    want_s, want_p = oracle.topk(x.astype(np.float64), k)
    for f in (tms.topk, tms.topk_split):
        ts, tp = f(s, co, k)
        torch.cuda.synchronize()
        ts, tp = ts.cpu().numpy()[0].astype(np.float64), tp.cpu().numpy()[0]
        assert np.array_equal(tp, want_p)
        assert ((ts == want_s) | (np.isnan(ts) & np.isnan(want_s))).all()


@pytest.mark.parametrize("k", [1, 17, 256])
@pytest.mark.parametrize("n", [1025, 4097, 20_481, 70_003])
def test_equal_scores_across_the_cut(cuda_lib, n, k):
    """Every list holds more equal scores than the survivor buffer: none above
    them, one fewer than k above them, and k above them (then none is taken)."""
    g = np.random.default_rng(n + k)
    for above in (0, k - 1, k):
        if above + 1025 > n:
            continue
        for tied in (2.0, -np.inf):
            x = np.full(n, tied, np.float32)
            rest = g.permutation(n)
            x[rest[:above]] = 3.0 + g.random(above).astype(np.float32)
            if tied == 2.0:
                x[rest[above + 1025:]] = -g.random(n - above - 1025).astype(np.float32)
            _check(x, k)
    _check(np.full(n, np.nan, np.float32), k)


@pytest.mark.parametrize("k", [10, 100])
@pytest.mark.parametrize("n", [20_000, 100_000])
def test_a_bound_that_many_keys_exceed(cuda_lib, n, k):
    """The largest scores all in the share of five warps, so that the bound is
    another warp's and thousands of distinct keys lie above it."""
    g = np.random.default_rng(n)
    x = g.random(n).astype(np.float32)
    x[np.arange(n) % 1024 < 160] += 5.0
    _check(x, k)


def test_equal_scores_cost_what_others_do(cuda_lib):
    """10,000 equal scores: 1.6 times a list of distinct ones (a selection
    that gives up on them and starts again digit by digit took 3.9 times)."""
    import torch
    from paper_2606_26439_gb300 import tms
    n = 10_000
    co = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    out = (torch.empty((1, 10), device="cuda"), torch.empty((1, 10), dtype=torch.int32, device="cuda"))
    t = []
    for s in (torch.randn(n, device="cuda"), torch.full((n,), 1.0, device="cuda")):
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(100):
                tms.topk(s, co, 10, *out)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        t.append(best)
    assert t[1] < 2.5 * t[0], t
