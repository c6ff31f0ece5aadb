"""Loads of kernels that start while the kernel before them still runs (launch_dependent, pdl_wait).

Behind the wait such a kernel reads what others have just written.  A read-only load (__ldg, or a pointer that the
compiler may treat alike: const __restrict__) promises that nobody writes the data while the kernel runs, and may be moved ahead
of the wait.  Whether it is moved cannot be seen from outputs, so the sources are held to the rule."""
import os
import re

import pytest

import paper_2503_16257_b200 as P

CSRC = os.path.join(os.path.dirname(os.path.abspath(P.__file__)), "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _functions(name):
    """(head, body) of every function of a source file, comments removed."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    text = re.sub(r"^\s*#(?:[^\n]*\\\n)*[^\n]*$", "", text, flags=re.M)
    found, at = [], 0
    while True:
        m = re.compile(r"\{").search(text, at)
        if not m:
            return found
        head = re.split(r"[;{}]", text[:m.start()])[-1]
        at = m.end()
        if "(" not in head or re.match(r"\s*(?:namespace|struct|template\s*<[^(]*>\s*struct|extern)\b", head):
            continue                                       # a scope that holds functions
        depth = 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        found.append((head, text[m.end():at]))


def test_the_scan_sees_the_kernels():
    waiting = [re.search(r"(\w+)\s*\(", h.split("__launch_bounds__")[-1].split(")", 1)[-1]).group(1) for f in FILES for h, b in _functions(f)
               if "__global__" in h and "pdl_wait()" in b]
    assert sorted(waiting) == ["decode_block_kernel", "decode_merge_kernel", "decode_stream_kernel", "decode_stream_stp_kernel",
                               "k_encode_kernel", "k_range_kernel", "v_quantize_kernel"]


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_load_behind_a_wait(name):
    functions = _functions(name)
    with_waits = name.endswith(".cuh") or any("__global__" in h and "pdl_wait()" in b for h, b in functions)
    for head, body in functions:
        if "__global__" not in head:                       # helpers run on either side of a wait
            assert not (with_waits and "__ldg" in body), head
        elif "pdl_wait()" in body:
            assert "__ldg" not in body.split("pdl_wait()", 1)[1], head
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", head), head
