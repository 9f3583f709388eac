"""Every kernel of the library waits before it touches global memory.

test_launch_sources finds the kernels by the names given to launch_dependent,
and does not see one that reaches it through a function's parameter (the E4M3
quantizer).  This goes by the definitions: every __global__ function but the
measurement probes, which are launched with <<<>>>, calls griddep_wait() and
uses none of its pointer arguments, nor a pointer in its argument struct,
before that.  Reads the CUDA sources as text; needs no GPU.
"""
from __future__ import annotations

import re

import pytest

from tests.test_launch_sources import _kernel_body, _sources

PROBES = {"lds_kernel", "read_kernel"}


def _kernels(text):
    """{name: (parameters, body)} of the __global__ definitions in `text`."""
    text = re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)", "", text)
    out = {}
    for m in re.finditer(r"__global__\s+void\s+(\w+)\s*\(([^{;]*)\)\s*\{", text):
        out[m.group(1)] = (m.group(2), _kernel_body(text, m.group(1)))
    return out


def _touched_early(parameters, body):
    """Names of global memory that the body mentions before its wait (all of
    them if it never waits)."""
    names = re.findall(r"\*\s*(?:__restrict__\s*)?(\w+)\s*(?:,|$)", parameters)
    wait = body.find("griddep_wait();")
    before = body[:wait] if wait >= 0 else body
    hit = {n for n in names if re.search(rf"(?<![.\w]){n}\b", before)}
    hit |= set(re.findall(r"\ba\.(out|lut|codes|offsets|lengths|cand_ids|cand_offsets|pq_codes|pq_codebook|q_scales|"
                          r"t_scales|err)\b", before))
    if "__ldg(" in before:
        hit.add("__ldg")
    return hit if wait >= 0 else hit | {"no wait"}


def test_every_kernel_waits_first():
    kernels = {}
    for text in _sources().values():
        kernels.update(_kernels(text))
    assert {"quantize_kernel", "dense_tc_kernel", "dense_f32_kernel", "score_kernel", "score_kernel_staged", "lut_kernel",
            "topk_kernel", "topk_slice_kernel", "topk_merge_kernel", "shortlist_csr", "shortlist_ids"} <= set(kernels)
    for name in sorted(set(kernels) - PROBES):
        assert not _touched_early(*kernels[name]), name


@pytest.mark.parametrize("name", ["quantize_kernel", "topk_slice_kernel", "score_kernel_staged"])
def test_a_missing_or_late_wait_is_seen(name):
    text = next(t for t in _sources().values() if name in _kernels(t))
    parameters, body = _kernels(text)[name]
    assert "no wait" in _touched_early(parameters, body.replace("griddep_wait();", ""))
    late = body.replace("griddep_wait();", "", 1).rstrip("}") + "griddep_wait(); }"
    assert _touched_early(parameters, late)


def test_plain_launches_are_only_the_probes():
    plain = set()
    for text in _sources().values():
        plain |= {m.group(1).split("::")[-1] for m in re.finditer(r"([A-Za-z_][\w:]*)(?:<[^<>]*>)?<<<", text)}
    assert plain == PROBES
