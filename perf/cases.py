"""The work a user of this library has it do, as measurable cases.

Each case is one call sequence of the public Python binding on inputs of a
passage-retrieval store: late-interaction MaxSim over candidate lists, dense
(fp16 / bf16 / fp32), FP8 and product-quantized, for per-query lists and for
queries that share one list, with the top-k that follows, the encoding of an
FP8 store, and the serving loop.  Sizes are those of the repository's
benchmark and tests, with odd and ragged ones among them.

``prepare`` builds what a program holds before the call (the store, the
lists, the query batch, its output buffers and top-k workspace), ``run`` is
one pass, ``exact`` the same outputs in 64 bits from plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_26439_gb300 import tms

DEV = "cuda"
TORCH_TYPE = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
ELEM = {"f16": 2, "bf16": 2, "f32": 4}
PQ_M, PQ_K = 16, 256


def listed():
    return [
        # One interactive query re-ranks the 1,000 passages of a first stage:
        # launches, latency and host calls count.
        _lists("rerank_f16_1x1000", "rerank", "f16", queries=1, cand=1000, docs=100_000),
        # One query over a small collection of fixed 128-token passages, top-10.
        _lists("rerank_f16_1x10000", "rerank", "f16", queries=1, cand=10_000, docs=10_000, lo=128, hi=128),
        # A batch of 16 queries, 100,000 candidates each, of a 500,000-document store.
        _lists("rerank_f16_16x100000", "rerank", "f16", queries=16, cand=100_000, docs=500_000),
        # The same step on an fp32 store.
        _lists("rerank_f32_4x20000", "rerank", "f32", queries=4, cand=20_000, docs=100_000),
        # Every query of a batch over one list, large token embeddings (dimension tiling).
        _shared("shared_bf16_32x20011_d768", "shared", "bf16", queries=32, cand=20_011, d=768),
        # The same at the usual dimension, with a query count that fills no group evenly.
        _shared("shared_f16_37x60000_d128", "shared", "f16", queries=37, cand=60_000, d=128),
        # Queries quantized and scored on the FP8 store, top-100 as a shortlist.
        _lists("rerank_fp8_16x20000", "rerank_fp8", "f16", queries=16, cand=20_000, docs=200_000, k=100),
        # A batch of queries over a whole FP8 store.
        _shared("shared_fp8_64x40009", "shared_fp8", "f16", queries=64, cand=40_009, d=128),
        # Per-query lists on a product-quantized store: table, score, top-10.
        _lists("rerank_pq_16x50000", "rerank_pq", "f16", queries=16, cand=50_000, docs=200_000, half_table=False),
        # A batch of queries over a whole product-quantized store, on the tensor cores.
        _shared("shared_pq_64x40000", "shared_pq", "f16", queries=64, cand=40_000, d=128),
        # The FP8 copy of a store is built from its fp16 tokens.
        {"name": "encode_fp8_4000037", "op": "encode_fp8", "dtype": "f16", "rows": 4_000_037, "d": 128},
        # A burst of requests to the serving loop: fp16 lists and FP8 lists with an fp16 re-score.
        {"name": "serve_48_requests", "op": "serve", "dtype": "f16", "requests": 48, "docs": 200_000,
         "min_list": 1000, "max_list": 20_000, "lo": 32, "hi": 180, "nq": 32, "d": 128, "k": 10, "rescore": 100},
    ]


def _lists(name, op, dtype, queries, cand, docs, lo=32, hi=180, nq=32, d=128, k=10, **more):
    return {"name": name, "op": op, "dtype": dtype, "queries": queries, "cand": cand, "docs": docs, "lo": lo,
            "hi": hi, "nq": nq, "d": d, "k": k, **more}


def _shared(name, op, dtype, queries, cand, d, lo=32, hi=180, nq=32):
    return {"name": name, "op": op, "dtype": dtype, "queries": queries, "cand": cand, "docs": cand, "lo": lo,
            "hi": hi, "nq": nq, "d": d}


# ------------------------------------------------------------------- draw

#: Multiply-adds of one pass (token pairs x dimension) a drawn case may have, by operation.
_LIMIT = {"rerank": 6e11, "rerank_fp8": 3e11, "rerank_pq": 2.5e11, "shared": 1.5e12, "shared_fp8": 1e12,
          "shared_pq": 1e12}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("rerank", "rerank", "rerank", "shared", "shared", "rerank_fp8", "shared_fp8", "rerank_pq",
                     "shared_pq", "encode_fp8", "serve"))
    if op == "encode_fp8":
        d = rng.choice((64, 96, 128, 256, 768))
        return {"op": op, "dtype": rng.choice(("f16", "bf16", "f32")), "rows": _log(rng, 1000, 5e8 // d), "d": d}
    if op == "serve":
        return {"op": op, "dtype": rng.choice(("f16", "bf16")), "requests": rng.randint(1, 48),
                "docs": rng.randint(40_000, 200_000), "min_list": 1000, "max_list": rng.randint(2000, 20_000),
                "lo": 32, "hi": 180, "nq": rng.choice((24, 32)), "d": 128, "k": rng.choice((10, 100)),
                "rescore": rng.choice((0, 100))}
    lo, hi = rng.choice(((32, 180), (32, 180), (128, 128), (1, 64), (100, 300)))
    pq, fp8 = op.endswith("pq"), op.endswith("fp8")
    dims = (128,) if pq else ((64, 128, 256, 768) if fp8 else (64, 96, 128, 256, 768))
    c = {"op": op, "dtype": "f16" if pq else rng.choice(("f16", "bf16")), "lo": lo, "hi": hi, "nq": 32,
         "d": rng.choice(dims)}
    if op.startswith("shared"):
        c["queries"] = rng.randint(2, 64)
        c["nq"] = rng.choice((32, 32, rng.randint(8, 32)))
        c["cand"] = _log(rng, 1000, 100_000)
    else:
        c["queries"] = _log(rng, 1, 16)
        c["nq"] = rng.choice((32, 32, rng.randint(8, 128)))
        c["cand"] = _log(rng, 1000, 100_000)
        c["k"] = rng.choice((10, 10, 100, 1000))
        if op == "rerank":
            c["dtype"] = rng.choice(("f16", "bf16", "f16", "bf16", "f32"))
        if op == "rerank_pq":
            c["half_table"] = rng.random() < 0.5
    pair = c["queries"] * c["nq"] * c["d"] * (lo + hi) / 2
    cap = _LIMIT[op] / (6 if c["dtype"] == "f32" else 1)
    if op == "rerank" and c["d"] * ELEM[c["dtype"]] * c["queries"] * (lo + hi) / 2 * c["cand"] > 4e10:
        cap = min(cap, 4e10 * c["nq"] / ELEM[c["dtype"]])
    c["cand"] = max(1000, min(c["cand"], int(cap / pair)))
    store = c["d"] * (lo + hi) / 2 * ELEM[c["dtype"]]
    most = max(c["cand"], int(1.3e10 / store))
    c["docs"] = c["cand"] if op.startswith("shared") else min(most, c["cand"] * rng.randint(1, 5))
    return c


# ---------------------------------------------------------------- prepare

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _unit_rows(g, rows, d, dtype):
    """L2-normalised Gaussian rows in the storage type."""
    out = torch.empty((rows, d), dtype=dtype, device=DEV)
    step = max(1, (1 << 29) // d)
    for r in range(0, rows, step):
        x = torch.randn((min(rows, r + step) - r, d), generator=g, device=DEV)
        x /= x.norm(dim=1, keepdim=True).clamp_min(1e-30)
        out[r:r + step] = x
    return out


def _lengths(g, case):
    n = torch.randint(case["lo"], case["hi"] + 1, (case["docs"],), generator=g, device=DEV)
    return (torch.cumsum(n, 0) - n).contiguous(), n.to(torch.int32)


def _e4m3(x):
    """E4M3 codes and scales of rows (scale = amax / 448, both divisions in fp32)."""
    x = x.float()
    amax = x.abs().amax(-1)
    s = amax / torch.full_like(amax, 448.0)
    y = torch.where(s.unsqueeze(-1) > 0, x / s.unsqueeze(-1), torch.zeros_like(x))
    return y.clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8), s


def _e4m3_store(tokens):
    codes = torch.empty(tokens.shape, dtype=torch.uint8, device=DEV)
    scales = torch.empty(tokens.shape[0], dtype=torch.float32, device=DEV)
    step = max(1, (1 << 28) // tokens.shape[1])
    for r in range(0, tokens.shape[0], step):
        codes[r:r + step], scales[r:r + step] = _e4m3(tokens[r:r + step])
    return codes, scales


def _topk_buffers(case, n_cand):
    q, k = case["queries"], case["k"]
    return {"top": (torch.empty((q, k), dtype=torch.float32, device=DEV),
                    torch.empty((q, k), dtype=torch.int32, device=DEV)),
            "workspace": torch.empty(max(16, tms.topk_workspace_size(q, k, n_cand)), dtype=torch.uint8, device=DEV)}


class _Server(tms.Server):
    """A serving loop that ends with the program's last reference to it."""

    def __del__(self):
        self.close()


def prepare(case, seed):
    op, s = case["op"], {"case": case}
    dtype = TORCH_TYPE[case["dtype"]]
    if op == "encode_fp8":
        g, rows, d = _gen(seed, 1), case["rows"], case["d"]
        s["x"] = _unit_rows(g, rows, d, dtype)
        s["codes"] = torch.empty((rows, d), dtype=torch.uint8, device=DEV)
        s["scales"] = torch.empty(rows, dtype=torch.float32, device=DEV)
        return s
    s["offsets"], s["lengths"] = _lengths(_gen(seed, 2), case)
    n_tokens = int(s["offsets"][-1] + s["lengths"][-1])
    g = _gen(seed, 3)
    if op.endswith("pq"):
        s["codebook"] = torch.randn((PQ_M, PQ_K, case["d"] // PQ_M), generator=g, device=DEV)
        s["codes"] = torch.randint(0, PQ_K, (n_tokens, PQ_M), generator=g, device=DEV, dtype=torch.uint8)
    else:
        s["tokens"] = _unit_rows(g, n_tokens, case["d"], dtype)
        if op.endswith("fp8") or op == "serve":
            s["codes"], s["scales"] = _e4m3_store(s["tokens"])
            if op != "serve":
                del s["tokens"]
    g = _gen(seed, 4)
    n_q = case["requests"] if op == "serve" else case["queries"]
    s["queries"] = _unit_rows(g, n_q * case["nq"], case["d"], dtype).view(n_q, case["nq"], case["d"])
    if op == "serve":
        return _prepare_serve(s, case, seed)
    if op.startswith("shared"):
        s["cand"] = torch.randperm(case["docs"], generator=g, device=DEV).to(torch.int32)
        s["out"] = torch.empty((n_q, case["cand"]), dtype=torch.float32, device=DEV)
    else:
        n = case["cand"]
        s["cand"] = torch.cat([torch.randperm(case["docs"], generator=g, device=DEV)[:n] for _ in range(n_q)]).to(
            torch.int32)
        s["list_offsets"] = torch.arange(n_q + 1, dtype=torch.int64, device=DEV) * n
        s["out"] = torch.empty(n_q * n, dtype=torch.float32, device=DEV)
        s.update(_topk_buffers(case, n_q * n))
    if op == "rerank_pq":
        s["table"] = torch.empty((n_q, case["nq"], PQ_M, PQ_K), dtype=torch.float32, device=DEV)
    if op.endswith("fp8"):
        s["q_codes"] = torch.empty(s["queries"].shape, dtype=torch.uint8, device=DEV)
        s["q_scales"] = torch.empty(s["queries"].shape[:-1], dtype=torch.float32, device=DEV)
    return s


def _prepare_serve(s, case, seed):
    r = np.random.default_rng([int(seed), 5])
    s["host_queries"] = s["queries"].cpu()
    lens = np.exp(r.uniform(math.log(case["min_list"]), math.log(case["max_list"]), case["requests"])).astype(int)
    s["lists"] = [r.integers(0, case["docs"], n).astype(np.int32) for n in lens]
    torch.cuda.synchronize()
    s["server"] = _Server(s["tokens"], s["offsets"], s["lengths"], case["nq"], case["k"], max_batch_requests=64,
                          max_batch_candidates=2_000_000, max_pending=4096, fp8=(s["codes"], s["scales"]),
                          rescore_k=case["rescore"])
    return s


def _store_of(i):
    """Requests alternate between the fp16 store and its FP8 copy."""
    return tms.TMS_STORE_FP8 if i % 2 else tms.TMS_STORE_DENSE


# -------------------------------------------------------------------- run

def run(s):
    case = s["case"]
    op = case["op"]
    if op == "encode_fp8":
        return list(tms.quantize_e4m3(s["x"], s["codes"], s["scales"]))
    if op == "serve":
        server = s["server"]
        tickets = [server.submit(s["host_queries"][i], ids, _store_of(i)) for i, ids in enumerate(s["lists"])]
        done = [server.wait(t) for t in tickets]
        return [np.stack([x[0] for x in done]), np.stack([x[1] for x in done])]
    docs = (s["offsets"], s["lengths"], s["cand"])
    if op.endswith("fp8"):
        tms.quantize_e4m3(s["queries"], s["q_codes"], s["q_scales"])
        fp8 = (s["q_codes"], s["q_scales"], s["codes"], s["scales"])
    if op == "shared":
        return tms.score_dense_shared(s["queries"], s["tokens"], *docs, out=s["out"])
    if op == "shared_fp8":
        return tms.score_fp8_shared(*fp8, *docs, out=s["out"])
    if op == "shared_pq":
        return tms.score_pq_tc_shared(s["queries"], s["codebook"], s["codes"], *docs, out=s["out"])
    if op == "rerank":
        tms.score_dense(s["queries"], s["tokens"], *docs, s["list_offsets"], out=s["out"])
    elif op == "rerank_fp8":
        tms.score_fp8(*fp8, *docs, s["list_offsets"], out=s["out"])
    else:
        tms.build_pq_lut(s["queries"], s["codebook"], out=s["table"])
        tms.score_pq(s["table"], s["codes"], *docs, s["list_offsets"], out=s["out"], f16_table=case["half_table"])
    top = tms.topk_split(s["out"], s["list_offsets"], case["k"], s["out"].numel(), *s["top"],
                         workspace=s["workspace"])
    return [s["out"], *top]


# ------------------------------------------------------------------- work

def work(case):
    op, d = case["op"], case["d"]
    if op == "encode_fp8":
        return {"bytes": case["rows"] * (d * ELEM[case["dtype"]] + d + 4), "flops": 3 * case["rows"] * d}
    mean = (case["lo"] + case["hi"]) / 2
    if op == "serve":
        span = math.log(case["max_list"] / case["min_list"])
        pairs = case["requests"] * (case["max_list"] - case["min_list"]) / span
        queries, row = case["requests"], d * ELEM[case["dtype"]]  # half the requests read FP8 rows
        read = _distinct(case["docs"], pairs / 2) * mean * (row + d + 4)
        return {"bytes": read + 4 * pairs, "flops": 2 * pairs * mean * case["nq"] * d}
    pairs, queries = case["queries"] * case["cand"], case["queries"]
    row = PQ_M if op.endswith("pq") else (d + 4 if op.endswith("fp8") else d * ELEM[case["dtype"]])
    lists = case["cand"] if op.startswith("shared") else pairs
    # every document that is in some list once, its 12 bytes of offset and length, the ids, the scores
    docs = min(case["docs"], lists) if op.startswith("shared") else _distinct(case["docs"], pairs, case["cand"])
    return {"bytes": docs * (mean * row + 12) + 4 * lists + 4 * pairs + queries * case["nq"] * d * ELEM[case["dtype"]],
            "flops": 2 * pairs * mean * case["nq"] * d}


def _distinct(docs, pairs, per_list=1):
    """Expected number of distinct documents in lists of `per_list` drawn without replacement."""
    return docs * (1 - (1 - min(1.0, per_list / docs)) ** (pairs / per_list))


# ------------------------------------------------------------------ exact

def exact(case, seed):
    op = case["op"]
    if op == "encode_fp8":
        if case["rows"] * case["d"] > 1e9:
            return None
        x = prepare(case, seed)["x"]
        step = 1 << 18
        return [None, torch.cat([x[r:r + step].double().abs().amax(1) / 448 for r in range(0, len(x), step)])]
    if work(case)["flops"] * case["hi"] / ((case["lo"] + case["hi"]) / 2) > 9e12:
        return None  # over about 20 seconds in 64 bits
    s = prepare(case, seed)
    if op == "serve":
        top = torch.full((case["requests"], case["k"]), -math.inf, dtype=torch.float64, device=DEV)
        for i, ids in enumerate(s["lists"]):
            ids = torch.from_numpy(ids).to(DEV)
            q = s["queries"][i:i + 1].double()
            if _store_of(i) == tms.TMS_STORE_FP8:
                qs = _decode(*_e4m3(s["queries"][i:i + 1]))
                score = _maxsim(s, qs, ids, lambda r: _decode(s["codes"][r], s["scales"][r]))[0]
                if case["rescore"]:
                    ids = ids[score.topk(min(case["rescore"], len(ids))).indices]
            if _store_of(i) == tms.TMS_STORE_DENSE or case["rescore"]:
                score = _maxsim(s, q, ids, lambda r: s["tokens"][r].double())[0]
            best = score.topk(min(case["k"], len(score))).values
            top[i, :len(best)] = best
        return [top, None]
    q = _decode(*_e4m3(s["queries"])) if op.endswith("fp8") else s["queries"].double()
    if op.endswith("pq"):
        flat, sub = s["codebook"].double(), torch.arange(PQ_M, device=DEV)
        rows = lambda r: flat[sub, s["codes"][r].long()].flatten(-2)  # noqa: E731
    elif op.endswith("fp8"):
        rows = lambda r: _decode(s["codes"][r], s["scales"][r])  # noqa: E731
    else:
        rows = lambda r: s["tokens"][r].double()  # noqa: E731
    if op.startswith("shared"):
        return _maxsim(s, q, s["cand"], rows)
    n = case["cand"]
    scores = torch.cat([_maxsim(s, q[i:i + 1], s["cand"][i * n:(i + 1) * n], rows)[0] for i in range(len(q))])
    best = torch.full((len(q), case["k"]), -math.inf, dtype=torch.float64, device=DEV)
    k = min(n, case["k"])
    best[:, :k] = scores.view(len(q), n).topk(k).values
    return [scores, best, None]


def _decode(codes, scales):
    return codes.view(torch.float8_e4m3fn).double() * scales.double().unsqueeze(-1)


def _maxsim(s, q, ids, rows):
    """Eq. 1 in 64 bits of queries q [n][nq][d] over the documents `ids`: [n][ids]."""
    n, nq, d = q.shape
    out = torch.empty((n, len(ids)), dtype=torch.float64, device=DEV)
    longest = int(s["lengths"].max())
    flat = q.reshape(n * nq, d).T.contiguous()
    step = max(1, int(5e8 // (longest * max(d, n * nq))))
    for c in range(0, len(ids), step):
        i = ids[c:c + step].long()
        at = torch.minimum(torch.arange(longest, device=DEV), s["lengths"][i].long().unsqueeze(1) - 1)
        sim = rows((s["offsets"][i].unsqueeze(1) + at).flatten()) @ flat  # a row past the end repeats the last one
        out[:, c:c + step] = sim.view(len(i), longest, n, nq).amax(1).sum(-1).T
    return out
