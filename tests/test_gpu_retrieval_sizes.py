"""The retrieval kernels at the edges of their splits, bit for bit against the
oracle: buffers that start at every offset from a 16-byte boundary, one
round of a single CTA and one position more, more candidates than a CTA keeps
ballots for, more matches than the ranking buffer holds, and (the index)
tiles, digits and passes of the sort at their edges."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import f32
from paper_2511_01282_gb300 import respec as rs
from test_gpu_index import _cuda, build_index, compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _buffers(rng, lens, V, k):
    tok_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tokens = rng.integers(0, V, int(tok_off[-1])).astype(np.int32)
    for b, t in enumerate(lens):
        a = int(tok_off[b])
        if t > 4 * k + 8:  # the key at both ends of the buffer and in between
            for q in [k - 1, t - 2 - k] + rng.integers(k, t - k, 3).tolist():
                tokens[a + q - k + 1:a + q + 1] = tokens[a + t - k:a + t]
    return tokens, tok_off


def _scan(tokens, tok_off, ks, scores, theta, top_c, span_len, pos_cap):
    B = len(tok_off) - 1
    z = lambda *shape: torch.full(shape, -7, dtype=torch.int32, device="cuda")  # noqa: E731
    out = dict(count=z(B), pos=z(B, pos_cap), sel_pos=z(B, top_c), sel_len=z(B, top_c), spans=z(B, top_c, span_len),
               n_sel=z(B), status=z(B))
    p = rs.params(theta_score=theta, top_c=top_c, span_len=span_len)
    rs.rs_match_scan(_cuda(tokens), _cuda(tok_off), B, _cuda(ks), None, _cuda(scores), p, pos_cap, out["count"], out["pos"],
                     out["sel_pos"], out["sel_len"], out["spans"], out["n_sel"], out["status"])
    torch.cuda.synchronize()
    ref = oracle.match_scan(tokens, tok_off, ks, scores, f32(theta), top_c, span_len, pos_cap, gate_ok=None)
    for key, got in out.items():
        assert (got.cpu().numpy() == ref[key]).all(), key
    return ref


@pytest.mark.parametrize("k", [1, 2, 3, 8])
@pytest.mark.parametrize("V", [3, 400])
def test_scan_alignments_and_round_edges(k, V):
    # request lengths of 1 mod 4 walk through every alignment; 4096 candidate
    # positions are the most one CTA takes alone
    rng = np.random.default_rng(100 * k + V)
    lens = [1, 5, 129, 8185, 16381, 8197, 16389, 33, 8193, 17, 20001, 4089, 4097, 4101]
    tokens, tok_off = _buffers(rng, lens, V, k)
    scores = rng.random(len(tokens)).astype(np.float32)
    scores[rng.random(len(tokens)) < 0.2] = 0.5
    for pos_cap in (0, 1, 700):
        _scan(tokens, tok_off, np.full(len(lens), k, np.int32), scores, 0.3, 3, 8, pos_cap)


def test_scan_beyond_the_kept_ballots():
    # 16 x 2048 rows x 128 positions = 4194304: the last rows are tested again
    # for their positions, which the capacity reaches only with few matches, and
    # for their scores when the buffer of matches overflows
    rng = np.random.default_rng(7)
    tokens, tok_off = _buffers(rng, [3, 4194304 + 70001], 50000, 2)
    scores = rng.random(len(tokens)).astype(np.float32)
    ref = _scan(tokens, tok_off, np.array([1, 1], np.int32), scores, 0.3, 8, 4, 300)
    assert 20 < ref["count"][1] < 300
    _scan(tokens, tok_off, np.array([0, 2], np.int32), scores, 0.3, 8, 4, 300)
    tokens = rng.integers(0, 60, 4194304 + 70001).astype(np.int32)
    _scan(tokens, np.array([0, len(tokens)], np.int64), np.array([1], np.int32), scores[:len(tokens)], 0.3, 8, 4, 100)


@pytest.mark.parametrize("B", [1, 4, 5, 7, 8, 9, 40])
def test_scan_cluster_forms(B):
    # as many requests as the GPU runs clusters of 16 at once (7): those, of which a
    # request of less than 131072 candidates uses 8; more: clusters of 8; more than 8
    # requests, or up to 32768 candidates: half the threads
    rng = np.random.default_rng(B)
    lens = rng.choice([40, 4090, 4101, 8197, 30001, 32760, 32775], B).tolist()
    lens[0], lens[-1] = 130000, 131200
    tokens, tok_off = _buffers(rng, lens, 30, 2)
    scores = rng.random(len(tokens)).astype(np.float32)
    _scan(tokens, tok_off, rng.integers(1, 4, B).astype(np.int32), scores, 0.3, 8, 8, 900)


@pytest.mark.parametrize("lens,V", [([1023, 1024, 1025, 0, 1], 300), ([4096, 0, 0, 4097], 1), ([524288 - 5, 5], 70000),
                                    ([524289], 511), ([70001] * 3, 512), ([3] * 700, 1 << 18), ([262143], 40000),
                                    ([0, 262144, 0], 40000), ([65535], 40000), ([0, 65536, 0], 40000),
                                    ([8388608], 1 << 17), ([8388609], 1 << 17), ([300001, 0, 280000, 3], 20000), ([9000] * 4, 1 << 17)])
def test_index_sort_edges(lens, V):
    # tiles of 1024 and 4096 keys (524288 tokens is the last total with small
    # tiles), one to four passes, with two of them from 65536 tokens on tiles cut
    # at the first digit (as long as a key's second digit and its position, 9 and
    # 23 bits of 8388608 tokens, fit one word), empty requests, ids that nothing holds
    rng = np.random.default_rng(len(lens) + V)
    tokens, tok_off = _buffers(rng, lens, max(V, 2), 1)  # V = 1: ids 0 and (foreign) 1
    scores = rng.random(len(tokens)).astype(np.float32)
    ks = rng.integers(1, 3, len(lens)).astype(np.int32)
    compare(tokens, tok_off, ks, None, scores, 0.3, 4, 8, 50, V)


@pytest.mark.parametrize("common", [4095, 4096, 4097, 40000, 4300000])
def test_index_query_of_a_common_token(common):
    # the key's last token fills one round of one CTA, one more, several rounds
    # of the cluster, and more than the ballots it keeps
    rng = np.random.default_rng(common)
    t = common + common // 3 + 100
    tokens = rng.integers(1, 1000, t).astype(np.int32)
    tokens[rng.permutation(t - 1)[:common]] = 0
    tokens[-1] = 0
    tok_off = np.array([0, t], np.int64)
    scores = rng.random(t).astype(np.float32)
    for k in (1, 3):
        compare(tokens, tok_off, np.array([k], np.int32), None, scores, 0.3, 8, 4, 5000, 1000)


@pytest.mark.parametrize("n", [1, 31, 32, 33])
def test_append_of_one_warp_and_more(n):
    # up to 32 new tokens are one warp's; many of one id, so that its bucket's
    # room ends inside the append, and the overflow list's last slots
    rng = np.random.default_rng(n)
    V = 50
    bufs = [rng.integers(0, V, 60).astype(np.int32), np.zeros(0, np.int32), rng.integers(0, V, 9).astype(np.int32)]
    tok_off = np.concatenate([[0], np.cumsum([len(x) for x in bufs])]).astype(np.int64)
    idx, total = build_index(np.concatenate(bufs), tok_off, V)
    status = torch.full((3,), -1, dtype=torch.int32, device="cuda")

    def grow(extra):
        nonlocal bufs, tok_off
        bufs = [np.concatenate([a, e]).astype(np.int32) for a, e in zip(bufs, extra)]
        tok_off = np.concatenate([[0], np.cumsum([len(x) for x in bufs])]).astype(np.int64)
        tokens = np.concatenate(bufs)
        rs.rs_match_index_append(_cuda(tokens), _cuda(tok_off), 3, V, total, idx, status)
        scores = rng.random(len(tokens)).astype(np.float32)
        for k in (1, 2):
            compare(tokens, tok_off, np.full(3, k, np.int32), None, scores, 0.3, 4, 8, 5000, V, idx=idx, t_total=total)
        return status.tolist()

    for _ in range(4):
        assert grow([np.where(rng.random(n) < 0.7, 7, rng.integers(0, V, n)), np.full(n, 3), rng.integers(-2, V + 2, n)]) == [0, 0, 0]
    # request 1's overflow list: filled up to its last n // 2 slots, then past them
    fill = 4096 + 2 - len(bufs[1]) - n // 2
    assert grow([[], np.full(fill, 3), []]) == [0, 0, 0]
    assert grow([[1], np.full(n, 3), []]) == [0, rs.RS_ST_TRUNCATED, 0]


@pytest.mark.parametrize("form", ["scan", "index"])
@pytest.mark.parametrize("B", [2, 9])
@pytest.mark.parametrize("share", [0.02, 0.12, 0.7])
def test_many_matches(form, B, share):
    # rows of 128 candidates with few and with many matches (a lane per row, then
    # row by row), more matches than are ranked at once (64), than a CTA's
    # buffer holds (512), equal scores among them, and a capacity inside a row
    rng = np.random.default_rng(int(100 * share) + B)
    lens = rng.choice([300, 3000, 9000, 40001], B).tolist()
    lens[0] = 40001
    tokens, tok_off = _buffers(rng, lens, 500, 1)
    tokens[rng.random(len(tokens)) < share] = 7
    tokens[tok_off[1:] - 1] = 7
    scores = rng.random(len(tokens)).astype(np.float32)
    scores[tok_off[1]:] = np.where(rng.random(len(tokens) - tok_off[1]) < 0.5, 0.75, scores[tok_off[1]:])
    ks = np.ones(B, np.int32)
    for pos_cap, theta in ((130, 0.3), (5000, 0.9)):
        if form == "scan":
            _scan(tokens, tok_off, ks, scores, theta, 5, 8, pos_cap)
        else:
            compare(tokens, tok_off, ks, None, scores, theta, 5, 8, pos_cap, 500)
