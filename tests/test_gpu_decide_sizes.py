"""rs_accept's decisions and the trigger's push at the edges of their words and
rounds, bit for bit against the oracle: trees of up to 256 nodes, chains and
model paths that cross 32-node words, positions selected twice, more accepted
nodes than the list holds, and requests of one round of rows and more."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import f32
from paper_2511_01282_gb300 import respec as rs
from test_gpu_index import _cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _tree(rng, model, chains):
    """Model nodes and chains interleaved in index order (each chain a path from the root)."""
    par, src, chn, tips = [-1], [0], [-1], [0] * len(chains)
    left = [("m", 0)] * model + [("c", c) for c, n in enumerate(chains) for _ in range(n)]
    models = [0]
    for kind, c in [left[i] for i in rng.permutation(len(left))]:
        i = len(par)
        if kind == "m":
            par.append(models[-1] if rng.random() < 0.8 else int(rng.choice(models)))
            models.append(i)
        else:
            par.append(tips[c])
            tips[c] = i
        src.append(1 if kind == "m" else 2)
        chn.append(-1 if kind == "m" else c)
    return np.array(par, np.int32), np.array(src, np.uint8), np.array(chn, np.int8)


@pytest.mark.parametrize("seed,accept", [(0, 0.7), (1, 0.97), (2, 1.0), (3, 0.9)])
@pytest.mark.parametrize("phi,m,acc_cap", [(2, 2, 64), (7, 0, 300), (40, 1, 5)])
def test_decisions_over_long_trees(seed, accept, phi, m, acc_cap):
    rng = np.random.default_rng(seed)
    V, top_c, beta = 96, 8, 5
    trees = [_tree(rng, 255, []), _tree(rng, 0, [255]), _tree(rng, 31, [32, 33, 64, 1]), _tree(rng, 0, []),
             _tree(rng, 100, [20] * 7), _tree(rng, 3, [31, 63, 95])]
    node_off = np.concatenate([[0], np.cumsum([len(t[0]) for t in trees])]).astype(np.int32)
    R, B = int(node_off[-1]), len(trees)
    par, src, chn = (np.concatenate([t[i] for t in trees]) for i in range(3))
    z = rng.standard_normal((R, V)).astype(np.float32)
    tok = rng.integers(0, V, R).astype(np.int32)
    for b in range(B):
        n0 = int(node_off[b])
        for i in range(n0 + 1, int(node_off[b + 1])):
            p = n0 + int(par[i])
            if rng.random() < accept:
                tok[i] = int(z[p].argmax())
            elif rng.random() < 0.8:
                tok[i] = int(np.argsort(-z[p])[rng.integers(1, 5)])
    t = 400
    tok_off = (np.arange(B + 1) * t).astype(np.int64)
    scores = rng.random(B * t).astype(np.float32)
    sel = rng.integers(-1, 40, (B, top_c)).astype(np.int32)  # often the same position twice
    sel[1, 0], sel[4, 2] = t + 3, 7                          # past the buffer, where the chain exists
    p = rs.params(beta=beta, tau=1.0, phi=phi, m=m, top_c=top_c)
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")  # noqa: E731
    flt = lambda n: torch.zeros(n, device="cuda")                         # noqa: E731
    o = dict(argmax=i32(R), topk=i32(R, beta), lse=flt(R), p_tok=flt(R), entropy=flt(R), acc_len=i32(B),
             acc_nodes=i32(B, acc_cap), bonus=i32(B), winner=i32(B), commit=torch.zeros(R, dtype=torch.uint8, device="cuda"),
             scores=_cuda(scores), status=i32(B))
    ws = torch.empty(rs.rs_accept_workspace_size(R, V, beta), dtype=torch.uint8, device="cuda")
    rs.rs_accept(_cuda(z), R, V, _cuda(node_off), B, _cuda(tok), _cuda(par), _cuda(src), _cuda(chn), _cuda(sel), _cuda(tok_off),
                 p, acc_cap, o["argmax"], o["topk"], o["lse"], o["p_tok"], o["entropy"], o["acc_len"], o["acc_nodes"], o["bonus"],
                 o["winner"], o["commit"], o["scores"], o["status"], ws)
    torch.cuda.synchronize()
    ref = oracle.accept(z, node_off, tok, par, src, chn, sel, tok_off, scores, beta, f32(1.0), phi, m, f32(p.alpha), acc_cap)
    for k in ("argmax", "topk", "acc_len", "acc_nodes", "bonus", "winner", "commit", "scores", "status"):
        assert (o[k].cpu().numpy() == ref[k]).all(), k
    assert (ref["status"] & rs.RS_ST_BAD_POS).any()


@pytest.mark.parametrize("V", [500, 8193])
def test_trigger_over_row_ranges(V):
    # a row per thread up to 256 rows of a request, more in rounds; rows of one
    # chunk (V <= 8192) need no merge
    rng = np.random.default_rng(V)
    l, n = 5, np.array([1, 255, 256, 257, 0, 600])
    B, R = len(n), int(n.sum())
    row_off = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    z = (rng.standard_normal((R, V)) * rng.uniform(0.5, 6, (R, 1))).astype(np.float32)
    for share in (0.0, 0.01, 0.5, 1.0):
        commit = (rng.random(R) < share).astype(np.uint8)
        hist, hist_n = rng.uniform(0.1, 3, (B, l)).astype(np.float32), rng.integers(0, l + 1, B).astype(np.int32)
        p = rs.params(l=l)
        h, hn = _cuda(hist), _cuda(hist_n)
        ent, hb = torch.zeros(R, device="cuda"), torch.zeros(B, device="cuda")
        ks, ok = torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.uint8, device="cuda")
        ws = torch.empty(max(256, rs.rs_entropy_gate_workspace_size(R, V)), dtype=torch.uint8, device="cuda")
        for rows in (False, True):  # the whole call, then the push alone on its entropies
            h.copy_(_cuda(hist))
            hn.copy_(_cuda(hist_n))
            if rows:
                rs.rs_entropy_gate_rows(ent, _cuda(row_off), _cuda(commit), B, p, h, hn, ks, hb, ok)
            else:
                rs.rs_entropy_gate(_cuda(z), R, V, _cuda(row_off), _cuda(commit), B, p, h, hn, ent, ks, hb, ok, ws)
            torch.cuda.synchronize()
            got = ent.cpu().numpy().astype(np.float64)
            assert np.abs(got - oracle.entropy_rows(z)).max() < 1e-3
            g = oracle.gate(got, row_off, commit, hist, hist_n, l, f32(p.lambda_e), f32(p.theta_entropy))
            assert (ks.cpu().numpy() == g["k_star"]).all() and (ok.cpu().numpy() == g["ok"]).all()
            assert (hb.cpu().numpy() == g["h_best"].astype(np.float32)).all() and (hn.cpu().numpy() == g["hist_n"]).all()
            for b in range(B):
                k = int(g["hist_n"][b])
                assert (h.cpu().numpy()[b, :k] == g["hist"].astype(np.float32)[b, :k]).all()
