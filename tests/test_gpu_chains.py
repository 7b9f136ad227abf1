"""Calls that feed one another on one stream with nothing in between: no copy, no
synchronisation and no other kernel, so that every call is launched while the one
whose outputs it reads may still run.  Whatever is handed over starts out as
poison (every row committed, entropies of 100 nats, every position selected), and
the score table and the histories are updated in place; the oracle replays the
whole chain afterwards."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import f32, host
from paper_2511_01282_gb300 import respec as rs
from test_gpu_decide_sizes import _tree
from test_gpu_index import _cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _batch(rng, B, V, top_c):
    """Trees of a batch and logits whose argmax is a child's token more often than not."""
    trees = [_tree(rng, int(rng.integers(1, 12)), rng.integers(1, 6, top_c).tolist()) for _ in range(B)]
    off = np.concatenate([[0], np.cumsum([len(t[0]) for t in trees])]).astype(np.int32)
    par, src, chn = (np.concatenate([t[i] for t in trees]) for i in range(3))
    R = int(off[-1])
    z = (rng.standard_normal((R, V)) * rng.uniform(0.5, 8, (R, 1))).astype(np.float32)
    tok = rng.integers(0, V, R).astype(np.int32)
    for b in range(B):
        for i in range(int(off[b]) + 1, int(off[b + 1])):
            if rng.random() < 0.8:
                tok[i] = int(z[off[b] + par[i]].argmax())
    return dict(z=z, off=off, par=par, src=src, chn=chn, tok=tok, R=R)


def _accept(c, d, B, V, sel, tok_off, p, cap, scores, ws):
    rs.rs_accept(d["z"], c["R"], V, d["off"], B, d["tok"], d["par"], d["src"], d["chn"], sel, tok_off, p, cap, d["argmax"], d["topk"],
                 d["lse"], d["p_tok"], d["entropy"], d["acc_len"], d["acc_nodes"], d["bonus"], d["winner"], d["commit"], scores,
                 d["status"], ws)


@pytest.mark.parametrize("retrieval", ["scan", "index"])
@pytest.mark.parametrize("B,V", [(3, 500), (2, 20000), (1, 70001)])  # rows of one chunk, of a cluster, merged by a kernel
def test_steps_without_a_wait(B, V, retrieval):
    rng = np.random.default_rng(V + B)
    steps, l, top_c, span, pos_cap, cap, t = 16 if V < 70000 else 6, 3, 3, 8, 32, 16, 4000
    p = rs.params(l=l, top_c=top_c, span_len=span, theta_entropy=2.0)
    tokens = rng.integers(0, 40, B * t).astype(np.int32)
    tok_off = (np.arange(B + 1) * t).astype(np.int64)
    scores = rng.random(B * t).astype(np.float32)
    hist, hist_n = np.zeros((B, l), np.float32), np.zeros(B, np.int32)
    d_tok, d_off, d_scores, d_hist, d_hist_n = (_cuda(a) for a in (tokens, tok_off, scores, hist, hist_n))
    full = lambda v, *s, dtype=torch.int32: torch.full(s, v, dtype=dtype, device="cuda")  # noqa: E731
    chain = []
    for _ in range(steps):
        two = []
        for _ in range(2):  # both trees of a step update the same table
            c = _batch(rng, B, V, top_c)
            d = {k: _cuda(c[k]) for k in ("z", "off", "par", "src", "chn", "tok")}
            R = c["R"]
            d.update(argmax=full(-7, R), topk=full(-7, R, p.beta), lse=full(0.0, R, dtype=torch.float32),
                     p_tok=full(0.0, R, dtype=torch.float32), entropy=full(100.0, R, dtype=torch.float32), acc_len=full(-7, B),
                     acc_nodes=full(-7, B, cap), bonus=full(-7, B), winner=full(-7, B), commit=full(1, R, dtype=torch.uint8),
                     status=full(-7, B))
            two.append((c, d))
        g = dict(k_star=full(1, B), h_best=full(0.0, B, dtype=torch.float32), ok=full(1, B, dtype=torch.uint8))
        s = dict(count=full(-7, B), pos=full(-7, B, pos_cap), sel_pos=full(5, B, top_c), sel_len=full(-7, B, top_c),
                 spans=full(-7, B, top_c, span), n_sel=full(-7, B), status=full(-7, B))
        chain.append((two, g, s))
    ws = torch.empty(max(rs.rs_accept_workspace_size(c["R"], V, p.beta) for two, _, _ in chain for c, _ in two), dtype=torch.uint8,
                     device="cuda")
    idx = torch.empty(rs.rs_match_index_bytes(B, 64, B * t), dtype=torch.uint8, device="cuda")
    rs.rs_match_index_build(d_tok, d_off, B, 64, B * t, idx)
    torch.cuda.synchronize()
    k_star, ok = full(2, B), full(1, B, dtype=torch.uint8)
    torch.cuda.synchronize()
    for two, g, s in chain:
        args = (d_tok, d_off, B, k_star, ok, d_scores, p, pos_cap, s["count"], s["pos"], s["sel_pos"], s["sel_len"], s["spans"],
                s["n_sel"], s["status"])
        if retrieval == "scan":
            rs.rs_match_scan(*args)
        else:
            rs.rs_match_scan_indexed(*args, 64, B * t, idx)
        for c, d in two:
            _accept(c, d, B, V, s["sel_pos"], d_off, p, cap, d_scores, ws)
        rs.rs_entropy_gate_rows(two[1][1]["entropy"], two[1][1]["off"], two[1][1]["commit"], B, p, d_hist, d_hist_n, g["k_star"],
                                g["h_best"], g["ok"])
        k_star, ok = g["k_star"], g["ok"]
    torch.cuda.synchronize()
    ks, kok = np.full(B, 2, np.int32), np.ones(B, np.uint8)
    for i, (two, g, s) in enumerate(chain):
        ref = oracle.match_scan(tokens, tok_off, ks, scores, f32(p.theta_score), top_c, span, pos_cap, gate_ok=kok)
        for key, got in s.items():
            assert (host(got) == ref[key]).all(), (i, key)
        for c, d in two:
            a = oracle.accept(c["z"], c["off"], c["tok"], c["par"], c["src"], c["chn"], ref["sel_pos"], tok_off, scores, p.beta,
                              f32(p.tau), p.phi, p.m, f32(p.alpha), cap)
            scores = a["scores"]
            for key in ("argmax", "topk", "acc_len", "acc_nodes", "bonus", "winner", "commit", "status"):
                assert (host(d[key]) == a[key]).all(), (i, key)
        H = host(two[1][1]["entropy"]).astype(np.float64)
        assert np.abs(H - oracle.entropy_rows(two[1][0]["z"])).max() < 1e-3
        o = oracle.gate(H, two[1][0]["off"], a["commit"], hist, hist_n, l, f32(p.lambda_e), f32(p.theta_entropy))
        hist, hist_n = o["hist"].astype(np.float32), o["hist_n"]
        ks, kok = o["k_star"], o["ok"]
        assert (host(g["k_star"]) == ks).all() and (host(g["ok"]) == kok).all() and (host(g["h_best"]) == o["h_best"].astype(np.float32)).all(), i
    assert (host(d_scores) == scores).all()
    assert (host(d_hist_n) == hist_n).all() and all((host(d_hist)[b, :n] == hist[b, :n]).all() for b, n in enumerate(hist_n))


@pytest.mark.parametrize("V", [500, 8193])  # rows of one chunk need no merge
def test_gates_on_one_history(V):
    rng = np.random.default_rng(V)
    B, l, calls, each = 5, 4, 40, 7
    R, p = B * each, rs.params(l=l)
    off = (np.arange(B + 1) * each).astype(np.int32)
    z = (rng.standard_normal((calls, R, V)) * rng.uniform(0.3, 6, (calls, R, 1))).astype(np.float32)
    commit = (rng.random((calls, R)) < 0.2).astype(np.uint8)
    hist, hist_n = np.zeros((B, l), np.float32), np.zeros(B, np.int32)
    d_z, d_off, d_commit, d_hist, d_hist_n = (_cuda(a) for a in (z, off, commit, hist, hist_n))
    ent = torch.full((calls, R), 100.0, device="cuda")
    ks, hb, ok = (torch.full((calls, B), 1, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.uint8))
    ws = torch.empty(max(256, rs.rs_entropy_gate_workspace_size(R, V)), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for i in range(calls):
        rs.rs_entropy_gate(d_z[i], R, V, d_off, d_commit[i], B, p, d_hist, d_hist_n, ent[i], ks[i], hb[i], ok[i], ws)
    torch.cuda.synchronize()
    for i in range(calls):
        H = host(ent[i]).astype(np.float64)
        assert np.abs(H - oracle.entropy_rows(z[i])).max() < 1e-3
        o = oracle.gate(H, off, commit[i], hist, hist_n, l, f32(p.lambda_e), f32(p.theta_entropy))
        hist, hist_n = o["hist"].astype(np.float32), o["hist_n"]
        assert (host(ks[i]) == o["k_star"]).all() and (host(ok[i]) == o["ok"]).all(), i
        assert (host(hb[i]) == o["h_best"].astype(np.float32)).all(), i
    assert (host(d_hist_n) == hist_n).all() and all((host(d_hist)[b, :n] == hist[b, :n]).all() for b, n in enumerate(hist_n))
