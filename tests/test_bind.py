"""The C++ marshalling of respec.py, without a GPU: which arguments it takes and
refuses.  The calls made here stop at the library's host checks."""
import ctypes

import pytest
import torch

from paper_2511_01282_gb300 import build


@pytest.fixture(scope="module")
def rs():
    build.build()
    from paper_2511_01282_gb300 import respec
    return respec


def _scan(rs, tokens=16, B=0, k_star=16, p=None, pos_cap=4, workspace=None, stream=0):
    rs.rs_match_scan(tokens, 16, B, k_star, None, 16, p or rs.params(), pos_cap, *([16] * 7), workspace, stream=stream)


def test_addresses_none_and_keywords_reach_the_library(rs):
    n = rs.rs_launch_count()
    _scan(rs)                                          # B = 0: nothing to do
    rs.rs_entropy_gate_rows(None, None, None, 0, rs.params(), None, None, None, None, None, stream=0)
    rs.rs_match_scan(tokens=16, tok_off=16, B=True - 1, k_star=16, gate_ok=None, scores=16, p=rs.params(), pos_cap=0,
                     count=16, pos=16, sel_pos=16, sel_len=16, spans=16, n_sel=16, status=16, stream=0)
    assert rs.rs_launch_count() == n


def test_parameters_arrive_whole(rs):
    for bad, word in ((dict(top_c=9), "top_c=9"), (dict(span_len=0), "span_len=0")):
        with pytest.raises(rs.RespecError, match=word) as e:
            _scan(rs, p=rs.params(**bad))
        assert e.value.status == rs.RS_ERR_INVALID_ARG
    with pytest.raises(rs.RespecError, match="lambda|l=0"):
        rs.rs_entropy_gate_rows(16, 16, 16, 0, rs.params(l=0), 16, 16, 16, 16, 16, stream=0)
    with pytest.raises(rs.RespecError, match="scale"):
        rs.rs_tree_verify_attn(16, 16, 16, 0, 16, 16, 16, 16, 1, 0, 4, 4, 64, -1.0, 16, 16, 16, None, stream=0)


def test_integers_wrap_as_in_c(rs):
    _scan(rs, B=1 << 32)                               # 0 in 32 bits
    with pytest.raises(rs.RespecError, match="negative B"):
        _scan(rs, B=(1 << 32) - 1)


@pytest.mark.parametrize("kw,err", [(dict(tokens=torch.zeros(4, dtype=torch.int32)), ValueError),
                                    (dict(tokens="text"), Exception), (dict(B=1.0), ctypes.ArgumentError),
                                    (dict(p=dict(l=3)), ctypes.ArgumentError), (dict(workspace=5), AttributeError),
                                    (dict(workspace=torch.zeros(4)), ValueError), (dict(stream="s"), AttributeError)])
def test_refused(rs, kw, err):
    with pytest.raises(err):
        _scan(rs, **kw)


def test_objects_with_a_tensors_attributes(rs):
    class Like:
        is_cuda, device = True, "like"

        def __init__(self, contiguous=True):
            self.c = contiguous

        def is_contiguous(self):
            return self.c

        def data_ptr(self):
            return 4096

        def numel(self):
            return 8

        def element_size(self):
            return 4

    _scan(rs, tokens=Like(), workspace=Like())
    with pytest.raises(ValueError, match="contiguous"):
        _scan(rs, tokens=Like(False))


@pytest.mark.gpu
def test_views_and_streams_on_the_gpu(rs):
    x = torch.arange(40, dtype=torch.int32, device="cuda")
    with pytest.raises(ValueError, match="contiguous"):
        _scan(rs, tokens=x[::2])
    out = {n: torch.zeros(s, dtype=torch.int32, device="cuda") for n, s in
           (("count", 1), ("pos", 4), ("sel_pos", 3), ("sel_len", 3), ("spans", 24), ("n_sel", 1), ("status", 1))}
    off, k = torch.tensor([0, 8], device="cuda"), torch.ones(1, dtype=torch.int32, device="cuda")
    scores = torch.full((8,), 0.5, device="cuda")
    tok = torch.tensor([9, 7, 1, 2, 7, 3, 4, 7], dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for stream in (None, side, side.cuda_stream, 0):
        for t in out.values():
            t.fill_(-7)
        torch.cuda.synchronize()
        rs.rs_match_scan(tok, off, 1, k, None, scores, rs.params(), 4, *out.values(), stream=stream)
        torch.cuda.synchronize()
        assert out["count"].tolist() == [2] and out["pos"].tolist() == [1, 4, -1, -1]
