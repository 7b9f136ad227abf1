"""Retrieval from the longest buffers that int32 positions reach, 2^31 - 1 tokens,
at every offset from a 16-byte boundary, and from one token more, which is
refused.  The matches are planted, so that the answer is known without a scan."""
import pytest
import torch

from paper_2511_01282_gb300 import respec as rs

pytestmark = [pytest.mark.gpu, pytest.mark.slow]
TOP = (1 << 31) - 1


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.fixture(scope="module")
def buffers():
    # 17 GB: tokens of zeros and scores of a half, both from a 16-byte boundary on
    yield torch.zeros(TOP + 8, dtype=torch.int32, device="cuda"), torch.full((TOP + 8,), 0.5, device="cuda")
    torch.cuda.empty_cache()


def _query(form, tok, sc, lead, t, k):
    """The outputs for one request of t tokens that begins `lead` tokens into the buffers."""
    off = torch.tensor([0, lead, lead + t], device="cuda")
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")  # noqa: E731
    o = dict(count=i32(2), pos=i32(2, 8), sel_pos=i32(2, 3), sel_len=i32(2, 3), spans=i32(2, 3, 4), n_sel=i32(2), status=i32(2))
    args = (tok, off, 2, torch.tensor([0, k], dtype=torch.int32, device="cuda"), None, sc, rs.params(top_c=3, span_len=4), 8, *o.values())
    if form == "scan":
        rs.rs_match_scan(*args)
    else:  # an index over the first 1000 tokens: the others are the linear tail, a candidate each
        first = torch.tensor([0, lead, lead + 1000], device="cuda")
        idx = torch.empty(rs.rs_match_index_bytes(2, 16, lead + 1000), dtype=torch.uint8, device="cuda")
        rs.rs_match_index_build(tok, first, 2, 16, lead + 1000, idx)
        rs.rs_match_scan_indexed(*args, 16, lead + 1000, idx)
    torch.cuda.synchronize()
    return {n: x[1].tolist() for n, x in o.items()}


@pytest.mark.parametrize("form", ["scan", "index"])
@pytest.mark.parametrize("lead", [0, 1, 2, 3])
def test_the_longest_buffer(buffers, form, lead):
    tok, sc = buffers
    t, k = TOP, 3
    ends = [k - 1, 700, 1 << 30, t - 133, t - 2 - k]
    where = [lead + p - i for p in ends + [t - 1] for i in (2, 1, 0)]
    at = torch.tensor(where, device="cuda")
    tok[at] = torch.tensor([7, 8, 9] * (len(ends) + 1), dtype=torch.int32, device="cuda")
    sc[lead + (1 << 30)] = 0.75
    got = _query(form, tok, sc, lead, t, k)
    tok[at] = 0
    sc[lead + (1 << 30)] = 0.5
    assert got["count"] == 5 and got["pos"] == ends + [-1] * 3 and got["status"] == 0 and got["n_sel"] == 3
    assert got["sel_pos"] == [1 << 30, t - 2 - k, t - 133] and got["sel_len"] == [4, 4, 4]
    assert got["spans"] == [[0] * 4, [0, 7, 8, 9], [0] * 4]


@pytest.mark.parametrize("form", ["scan", "index"])
def test_a_longer_buffer_is_refused(buffers, form):
    tok, sc = buffers
    none = dict(count=0, pos=[-1] * 8, sel_pos=[-1] * 3, sel_len=[0] * 3, spans=[[-1] * 4] * 3, n_sel=0)
    assert _query(form, tok, sc, 3, TOP + 1, 3) == dict(none, status=rs.RS_ST_TOO_LARGE)
    assert _query(form, tok, sc, 3, TOP + 1, 0) == dict(none, status=0)  # nothing to look for
