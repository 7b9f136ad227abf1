"""Rules of the CUDA sources that no run would show to be broken: whether a load
is moved above a kernel's wait for its predecessor is the compiler's choice, and
a stale value needs the two kernels to meet at the wrong moment."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_01282_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _text(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _span(s, at, pair):
    """The text between the pair of brackets that opens at or after `at`, and where it ends."""
    a = s.index(pair[0], at)
    depth = 0
    for i in range(a, len(s)):
        depth += (s[i] == pair[0]) - (s[i] == pair[1])
        if depth == 0:
            return s[a + 1:i], i
    raise AssertionError("unbalanced " + pair)


def _kernels():
    """(file, kernel, parameters, body) of every kernel."""
    out = []
    for f in SOURCES:
        s = _text(f)
        for m in re.finditer(r"__global__\s+void\b", s):
            at = m.end()
            while True:  # attributes with arguments, then the name
                w = re.compile(r"\s*(\w+)\s*\(").match(s, at)
                args, end = _span(s, at, "()")
                if not w.group(1).startswith("__"):
                    break
                at = end + 1
            body, _ = _span(s, end, "{}")
            out.append((f, w.group(1), args, body))
    return out


def _read_only(args):
    return re.findall(r"const\s+[^,()]*\*\s*__restrict__\s+(\w+)", args)


def test_every_kernel_is_found():
    names = {k for _, k, _, _ in _kernels()}
    assert {"gate_push", "accept_decide", "sample_walk", "attn_prep", "attn_tc_kernel", "index_query", "cut_scatter"} <= names
    assert len(names) >= 20


@pytest.mark.parametrize("kernel", [k for k in _kernels()], ids=lambda k: k[1])
def test_kernels_that_work_before_their_wait_have_plain_inputs(kernel):
    # a load through `const __restrict__` may be moved above the wait; with code
    # there the compiler has a place to move it to
    f, name, args, body = kernel
    before = re.split(r"pdl_enter\(\)|pdl_wait_prev\(\)", body)[0]
    early = re.sub(r"pdl_launch_next\(\)|[;\s]", "", before)
    assert "pdl_" in body, "%s neither waits for its predecessor nor says why" % name
    assert not early or not _read_only(args), "%s (%s): %s" % (name, f, _read_only(args))
