"""Kernels launched ahead of their predecessor's end (launch_chained): the rules
that make what they read safe, checked in the sources.

A chained kernel runs while kernels before it on the stream still write.  So
  - its first statement is chained(), which waits for them;
  - none of its pointers is __restrict__ (and nothing is read with __ldg): such a
    pointer promises that nobody else writes the data while the kernel runs, and
    the compiler may read through the non-coherent cache, or before the wait.
"""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2506_12727_gb300" / "csrc"


def _code():
    texts = [re.sub(r"//[^\n]*", "", f.read_text()) for f in sorted(CSRC.glob("*.cu*"))]
    return "\n".join(texts)


def _balanced(text, at, pair):
    """The text between the bracket at `at` and its partner, and where that lies."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return text[at + 1:i], i
    raise AssertionError("unbalanced")


def _kernels(code):
    """{name: (parameters, body)} of every __global__ function."""
    out = {}
    for m in re.finditer(r"__global__ void", code):
        at = m.end()
        head = re.match(r"\s*__launch_bounds__\s*", code[at:])
        if head:
            _, close = _balanced(code, at + head.end(), "()")
            at = close + 1
        name = re.match(r"\s*(\w+)\s*", code[at:])
        params, close = _balanced(code, at + name.end(), "()")
        body, _ = _balanced(code, code.index("{", close), "{}")
        out[name.group(1)] = (params, body)
    return out


CODE = _code()
KERNELS = _kernels(CODE)
CHAINED = sorted(set(re.findall(r"launch_chained\(\s*(\w+)", CODE)) - {"void"})


def test_the_chain_is_found():
    assert len(CHAINED) >= 20 and set(CHAINED) <= set(KERNELS)
    assert {"rs_downsweep", "preprocess_kernel", "bin_place_kernel", "set_counts_kernel"} <= set(CHAINED)


@pytest.mark.parametrize("name", CHAINED)
def test_a_chained_kernel_waits_first_and_reads_coherently(name):
    params, body = KERNELS[name]
    assert body.split(";")[0].strip() == "chained()"
    assert "__restrict__" not in params
    assert "__restrict__" not in body and "__ldg" not in body and ".nc" not in body
