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


def test_every_kernel_is_found():
    names = {k for _, k, _, _ in _kernels()}
    assert {"gate_push", "accept_decide", "sample_walk", "attn_prep", "attn_tc_kernel", "index_query", "cut_scatter"} <= names
    assert len(names) >= 20


@pytest.mark.parametrize("kernel", _kernels(), ids=lambda k: k[1])
def test_kernels_wait_for_their_predecessor(kernel):
    _, name, _, body = kernel
    assert re.search(r"\bpdl_(enter|wait_prev)\(\)|\bmat_enter\(", body), name


@pytest.mark.parametrize("name", SOURCES)
def test_loads_stay_behind_the_wait(name):
    # a load through a __restrict__ pointer (or __ldg) may be moved above the wait
    # for the kernel before, which may still be writing what is read; inlined, the
    # parameters of device functions are as good as the kernel's
    assert not re.findall(r"__restrict__|__ldg\b", _text(name))


def test_shared_structs_read_as_16_byte_words_are_aligned():
    # &sh.member as uint4: the struct's own alignment has to carry it, not what
    # else the kernel happens to keep in shared memory
    seen = 0
    for f in SOURCES:
        s = _text(f)
        for var, member in re.findall(r"reinterpret_cast<(?:const )?(?:u?int4|float4) \*>\(&(\w+)\.(\w+)", s):
            for struct in set(re.findall(r"(\w+)<[^<>]*>\s*&%s\b" % var, s)):
                assert re.search(r"struct\s+alignas\(16\)\s+%s\b" % struct, s), (f, struct)
                assert re.search(r"offsetof\(\w+, %s\) %% 16 == 0" % member, s), (f, struct, member)
                seen += 1
    assert seen >= 2
