"""Kernels that start before the launch ahead of them has completed read what that launch writes by ordinary loads.

The read-only path (__ldg, or a `const ... __restrict__` parameter, for which the compiler may take it) is for memory that
nobody writes while the kernel runs.  A programmatic dependent is resident while its predecessors still write, and such a load
is not held behind griddepcontrol.wait by anything.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_12335_b200", "csrc")
# What is complete before the kernel starts: the value norms' kernel and the fp32 pass 2 follow a pass that has waited itself
# before it lets them start, unless the caller's normalisers stand in for that pass; the large tiles are no dependents then.
COMPLETE = {"prefill_tc.cu": ["if (GIVEN) raw[j] = load_behind_wait(from); else raw[j] = __ldg(from);"],
            "prefill_simt.cu": ["template <typename T, int M> using Input = std::conditional_t<M == 8, const T* __restrict__, const T*>;"]}


def test_large_fp32_tiles_without_a_pass_before_them_are_launched_ordinarily():
    assert "if (M == 8 && lse_given) c2.attr[0].val.programmaticStreamSerializationAllowed = 0;" in _code("prefill_simt.cu")


def _code(name):
    """The file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _block(text, at, opening, closing):
    """The text from the first `opening` at or after `at` to the one that closes it."""
    begin = text.index(opening, at)
    depth = 0
    for i in range(begin, len(text)):
        depth += (text[i] == opening) - (text[i] == closing)
        if depth == 0:
            return text[begin:i + 1]
    raise AssertionError("unbalanced " + opening)


def _dependent_kernels(text):
    """(name, parameters, body) of the kernels that wait for the launch before them."""
    found = []
    for m in re.finditer(r"__global__\s+void\s*", text):
        at = m.end()
        if text.startswith("__launch_bounds__", at):
            at = text.index("(", at)
            at += len(_block(text, at, "(", ")"))
        name = re.compile(r"\s*(\w+)\s*(?=\()").match(text, at)
        at = name.end()
        params = _block(text, at, "(", ")")
        body = _block(text, at + len(params), "{", "}")
        if "griddepcontrol.wait" in body:
            found.append((name.group(1), params, body))
    return found


@pytest.mark.parametrize("name,kernels", [
    ("prefill_simt.cu", {"rowstats_kernel", "colsum_kernel"}),
    ("prefill_tc.cu", {"prefill_tc_kernel", "attention_fwd_tc_kernel", "reset_counters_kernel", "vnorm_kernel", "window_ring_tc_kernel"}),
    ("select.cu", {"select_kernel", "select_cluster_kernel"}),
    ("compact.cu", {"compact_kernel"}),
    ("window_ring.cu", {"window_ring_fma_kernel"}),
    ("decode_gqa.cu", {"group_mean_kernel"}),
    ("decode.cu", {"decode_kernel"}),
    ("decode_mma.cu", {"decode_mma_kernel"}),
])
def test_dependents_read_by_ordinary_loads(name, kernels):
    text = _code(name)
    found = _dependent_kernels(text)
    assert {k for k, _, _ in found} == kernels
    for kernel, params, _ in found:
        read_only = re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__", params)
        assert not read_only, (kernel, read_only)
    for f in (name, "simt_tile.cuh", "vatp_internal.cuh"):
        code = _code(f)
        for known in COMPLETE.get(f, ()):
            assert code.count(known) == 1
            code = code.replace(known, "")
        assert "__ldg" not in code and "ld.global.nc" not in code, f
        assert not re.search(r"(using|typedef).*__restrict__", code), f
