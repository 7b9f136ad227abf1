"""The workloads this library is timed on: its calls, as a decoding loop makes them.

A case is one call (or one short sequence of calls) of the public entry points, at a size that a serving program meets:

  attn    ``rs_tree_verify_attn`` of one layer: the draft trees of a batch against its bf16 KV cache
  gate    ``rs_entropy_gate``: the trigger, from the verify pass's logits
  accept  ``rs_accept``: row statistics, acceptance, score update, row entropies
  sample  ``rs_tree_sample``: lossless sampling verification of the model drafts
  scan    ``rs_match_scan``: retrieval from the token buffers
  index   ``rs_match_index_build`` over the prompts, then steps of ``rs_match_index_append`` + ``rs_match_scan_indexed``
  step    one whole ``VerifyStep``: eager calls, or replayed from a CUDA graph

Inputs follow ``synth/workloads.py`` (the same structure and distributions), drawn on the GPU from the seed.  Token buffers are
either uniform over the vocabulary, as there, or log-uniform ("zipf"), the frequency law of natural text, where the key's last
token is often a very common one.
"""
import math

import numpy as np
import torch

from paper_2511_01282_gb300 import respec as rs
from paper_2511_01282_gb300.pipeline import VerifyStep

POS_CAP = 1024  # match positions kept per request, as the workloads have it
ACC_CAP = 64


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest call there is: one short request, every call eager.  Launches and host time are all of it.
        dict(name="step-tiny", path="step", B=1, Hq=4, Hkv=4, D=64, ctx_lo=256, ctx_hi=256, model=4, chains=1, chain_len=4, V=1024,
             text="uniform", top_c=3, graph=False),
        # One interactive user of a 7B-shaped model: the steady-state step, replayed from a graph as a decoding loop does.
        dict(name="step-7b", path="step", B=1, Hq=32, Hkv=32, D=128, ctx_lo=2048, ctx_hi=2048, model=16, chains=3, chain_len=8,
             V=32000, text="uniform", top_c=3, graph=True),
        # Long-context retrieval-heavy verify with grouped-query heads: the attention that is bound by arithmetic.
        dict(name="attn-gqa16k", path="attn", B=1, Hq=32, Hkv=8, D=128, ctx_lo=16384, ctx_hi=16384, model=16, chains=8, chain_len=16),
        # Batched serving, ragged contexts and trees.
        dict(name="attn-batched", path="attn", B=16, Hq=32, Hkv=8, D=128, ctx_lo=1024, ctx_hi=8192, model=28, chains=2, chain_len=8),
        # The largest KV cache: four 32K-token requests of a 13B-shaped model.
        dict(name="attn-13b32k", path="attn", B=4, Hq=40, Hkv=40, D=128, ctx_lo=32768, ctx_hi=32768, model=32, chains=4, chain_len=8),
        # The trigger from the logits themselves (first step, or a loop without rs_accept's entropies), batched serving.
        dict(name="gate-batched", path="gate", B=16, nodes=45, V=128256),
        # Acceptance for four requests, 32K vocabulary ...
        dict(name="accept-13b", path="accept", B=4, nodes=65, chains=4, chain_len=8, V=32000, top_c=4),
        # ... and for one long retrieval-heavy tree at a 128K vocabulary.
        dict(name="accept-gqa16k", path="accept", B=1, nodes=145, chains=8, chain_len=16, V=128256, top_c=8),
        # Non-greedy decoding of one request at temperature 1.
        dict(name="sample-gqa16k", path="sample", B=1, nodes=145, chains=8, chain_len=16, V=128256, temperature=1.0),
        # Retrieval by scanning long token buffers (agents, long documents).
        dict(name="scan-256k", path="scan", B=4, tokens=262144, V=32000, text="zipf", top_c=3, span=8, k=2),
        # Retrieval by index: the index is built over the prompts, then eight decoding steps append to it and query it.
        dict(name="index-32k", path="index", B=4, tokens=32768, V=32000, text="uniform", top_c=4, span=8, k=3, steps=8, append=5),
        # The same over a million tokens per request, with the token frequencies of natural text.
        dict(name="index-1m", path="index", B=4, tokens=1048576, V=32000, text="zipf", top_c=3, span=8, k=2, steps=4, append=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng):
    """A model's vocabulary (some of the common sizes are odd), or any size."""
    return rng.choice([32000, 32001, 50257, 128256, 151936]) if rng.random() < 0.5 else _log_int(rng, 1000, 152000)


def _tree_shape(rng, most=200):
    chains = rng.randint(0, 8)
    chain_len = rng.choice([4, 8, 13, 16])
    model = _log_int(rng, 1, 64)
    while 1 + model + chains * chain_len > most:
        chains -= 1
    return dict(model=model, chains=chains, chain_len=chain_len)


def draw(rng):
    path = rng.choice(["attn", "attn", "attn", "gate", "accept", "accept", "sample", "scan", "index", "step"])
    if path == "attn":
        while True:
            Hkv, G = rng.choice([2, 4, 8, 16, 32, 40]), rng.choice([1, 2, 3, 4, 7, 8])
            hi = _log_int(rng, 64, 32768)
            c = dict(path=path, B=_log_int(rng, 1, 32), Hq=Hkv * G, Hkv=Hkv, D=rng.choice([64, 128, 128]),
                     ctx_lo=max(1, int(hi * rng.choice([1.0, 0.125]))), ctx_hi=hi, **_tree_shape(rng))
            if Hkv * G <= 64 and c["B"] * hi * Hkv * c["D"] * 4 <= 2.0e9 and work(c)["flops"] <= 1.0e11:
                return c
    if path == "gate":
        while True:
            c = dict(path=path, B=_log_int(rng, 1, 32), nodes=rng.randint(2, 96), V=_vocab(rng))
            if work(c)["bytes"] <= 4e8:
                return c
    if path in ("accept", "sample"):
        while True:
            t = _tree_shape(rng)
            c = dict(path=path, B=_log_int(rng, 1, 16), nodes=1 + t["model"] + t["chains"] * t["chain_len"], chains=t["chains"],
                     chain_len=t["chain_len"], V=_vocab(rng))
            if path == "accept":
                c["top_c"] = max(1, t["chains"])
            else:
                c["temperature"] = rng.choice([0.6, 0.8, 1.0, 1.3])
            if c["B"] * c["nodes"] * c["V"] * 4 <= 4e8:
                return c
    if path == "scan":
        tokens = _log_int(rng, 500, 1500000)
        return dict(path=path, B=rng.randint(1, max(1, min(16, 6000000 // tokens))), tokens=tokens, V=_vocab(rng),
                    text=rng.choice(["uniform", "zipf"]), top_c=rng.randint(1, 8), span=rng.choice([4, 8, 16]), k=rng.randint(1, 4))
    if path == "index":
        tokens = _log_int(rng, 4000, 1048576)
        return dict(path=path, B=rng.randint(1, max(1, min(16, 4194304 // tokens))), tokens=tokens, V=_vocab(rng),
                    text=rng.choice(["uniform", "zipf"]), top_c=rng.randint(1, 8), span=rng.choice([4, 8, 16]), k=rng.randint(1, 4),
                    steps=rng.randint(1, 4), append=rng.randint(1, 9))
    while True:
        Hkv, G = rng.choice([4, 8, 32]), rng.choice([1, 2, 4])
        hi = _log_int(rng, 64, 4096)
        t = _tree_shape(rng, 100)
        c = dict(path=path, B=_log_int(rng, 1, 8), Hq=Hkv * G, Hkv=Hkv, D=rng.choice([64, 128]), ctx_lo=max(40, hi // 2), ctx_hi=max(64, hi),
                 **t, V=_log_int(rng, 1000, 50000), text="uniform", top_c=max(1, t["chains"]), graph=rng.random() < 0.5)
        if Hkv * G <= 64 and work(c)["bytes"] <= 2e8:
            return c


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _lengths(case, seed):
    """Context length of every request, ragged between ctx_lo and ctx_hi."""
    return np.random.default_rng([seed, 1]).integers(case["ctx_lo"], case["ctx_hi"], size=case["B"], endpoint=True).astype(np.int32)


def _trees(B, model, chains, chain_len, V, seed):
    """The draft trees of a batch: root, a model tree that is bushiest near the root, then retrieved chains from the root."""
    g = np.random.default_rng([seed, 2])
    parents, source, chain = [], [], []
    for _ in range(B):
        par, src, chn = [-1], [0], [-1]
        for i in range(1, model + 1):
            par.append(int(i * g.random() ** 2))
            src.append(1)
            chn.append(-1)
        for c in range(chains):
            prev = 0
            for _ in range(chain_len):
                par.append(prev)
                src.append(2)
                chn.append(c)
                prev = len(par) - 1
        parents.append(par)
        source.append(src)
        chain.append(chn)
    N = 1 + model + chains * chain_len
    # children of one node carry different tokens, as a top-w expansion gives them
    tokens = (g.integers(0, V, size=(B, 1)) + np.arange(N) * max(1, V // N - 1)) % V
    return dict(N=N, node_off=(np.arange(B + 1) * N).astype(np.int32), parents=np.array(parents, np.int32).reshape(-1),
                source=np.array(source, np.uint8).reshape(-1), chain=np.array(chain, np.int8).reshape(-1),
                tree_tokens=tokens.astype(np.int32).reshape(-1))


def _logits(tree, V, gen):
    """[R, V] fp32 verify logits: normals with a per-row inverse temperature (row entropies of about 0.1 to 8 nats); of every
    parent's children some carry the row's best token and some one close to it."""
    parents, tokens = torch.from_numpy(tree["parents"]).cuda().long(), torch.from_numpy(tree["tree_tokens"]).cuda().long()
    R = parents.numel()
    z = torch.randn(R, V, device="cuda", generator=gen)
    lo, hi = math.log(math.sqrt(max(2.0 * (math.log(V) - 8.0), 0.25))), math.log(40.0)
    z *= torch.exp(lo + (hi - lo) * torch.rand(R, 1, device="cuda", generator=gen))
    top = z.max(dim=1).values
    kids = torch.nonzero(parents >= 0).squeeze(1)
    if kids.numel():
        rows = parents[kids] + (kids // tree["N"]) * tree["N"]
        kind = torch.rand(kids.numel(), device="cuda", generator=gen)
        order = torch.rand(kids.numel(), device="cuda", generator=gen)
        best = torch.full((R,), -1.0, device="cuda").scatter_reduce(0, rows, torch.where(kind < 0.6, order, -1.0), "amax")
        greedy = (kind < 0.6) & (order == best[rows])
        close = ~greedy & (kind < 0.8)
        raised = top[rows] + 0.1 + 0.9 * torch.rand(kids.numel(), device="cuda", generator=gen)
        near = top[rows] - 3.0 * torch.rand(kids.numel(), device="cuda", generator=gen)
        z[rows[close], tokens[kids[close]]] = near[close]
        z[rows[greedy], tokens[kids[greedy]]] = raised[greedy]
    return z


def _tokens(case, seed, B, t):
    """[B, t] token buffers: fresh tokens with copied 32-token spans (30 %); the trailing 4 tokens recur at eight places."""
    gen = _generator(seed * 4 + 1)
    V = case["V"]
    u = torch.rand(B, t, device="cuda", generator=gen)
    X = (torch.exp(u * math.log(V)) - 1).floor().clamp_(0, V - 1) if case["text"] == "zipf" else (u * V).floor().clamp_(0, V - 1)
    X = X.to(torch.int32)
    span = 32
    n = t // span
    if n > 1:
        copied = torch.rand(B, n, device="cuda", generator=gen) < 0.3
        src = (torch.rand(B, n, device="cuda", generator=gen) * torch.arange(n, device="cuda") * span).long()
        at = torch.arange(n, device="cuda") * span
        src = torch.where(copied, src, at)
        idx = (src[:, :, None] + torch.arange(span, device="cuda")).reshape(B, n * span)
        X[:, : n * span] = X.gather(1, idx)
    if t > 64:
        places = (8 + torch.rand(B, 8, device="cuda", generator=gen) * (t - 48)).long()
        for i in range(4):
            X.scatter_(1, places + i, X[:, t - 4 + i: t - 3 + i].expand(B, 8))
    return X


def _scores(n, gen):
    """The feedback table: S0 = 0.5, a third of the positions moved by feedback."""
    s = torch.rand(n, device="cuda", generator=gen)
    return torch.where(torch.rand(n, device="cuda", generator=gen) < 0.3, s, torch.full_like(s, 0.5))


def _history(B, l, seed):
    g = np.random.default_rng([seed, 3])
    return g.uniform(0.05, 3.0, size=(B, l)).astype(np.float32), g.integers(0, l, size=B, endpoint=True).astype(np.int32)


def _zeros(*shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def _scratch(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _attn_inputs(case, seed):
    B, Hq, Hkv, D = case["B"], case["Hq"], case["Hkv"], case["D"]
    tree = _trees(B, case["model"], case["chains"], case["chain_len"], case.get("V", 1 << 15), seed)
    ctx = _lengths(case, seed)
    rows = ctx.astype(np.int64) + tree["N"]
    kv_off = np.concatenate([[0], np.cumsum(rows)[:-1]]).astype(np.int64)
    gen = _generator(seed * 4)
    normal = lambda *s: torch.randn(*s, device="cuda", generator=gen, dtype=torch.bfloat16)  # noqa: E731
    R, T = B * tree["N"], int(rows.sum())
    return dict(tree=tree, ctx=ctx, kv_off=kv_off, R=R, T=T, q=normal(R, Hq, D), k=normal(T, Hkv, D), v=normal(T, Hkv, D))


def prepare(case, seed):
    return globals()["_prepare_" + case["path"]](case, seed)


def _prepare_attn(case, seed):
    x = _attn_inputs(case, seed)
    B, Hq, Hkv, D, R = case["B"], case["Hq"], case["Hkv"], case["D"], x["R"]
    out, lse, status = _zeros(R, Hq, D, dtype=torch.float32), _zeros(R, Hq, dtype=torch.float32), _zeros(B)
    ws = _scratch(rs.rs_tree_verify_attn_workspace_size(B, R, Hq, Hkv, D))
    args = (x["q"], x["k"], x["v"], x["T"], _cuda(x["kv_off"]), _cuda(x["ctx"]), _cuda(x["tree"]["node_off"]),
            _cuda(x["tree"]["parents"]), B, R, Hq, Hkv, D, D ** -0.5, out, lse, status, ws)
    return dict(call=rs.rs_tree_verify_attn, args=args, out=dict(out=out, lse=lse, status=status))


def _prepare_gate(case, seed):
    B, V = case["B"], case["V"]
    tree = _trees(B, case["nodes"] - 1, 0, 0, V, seed)
    logits = _logits(tree, V, _generator(seed * 4))
    p = rs.params()
    R = B * tree["N"]
    commit = (np.random.default_rng([seed, 4]).random(R) < 0.1).astype(np.uint8)
    commit[:: tree["N"]] = 1
    hist, hist_n = (_cuda(a) for a in _history(B, p.l, seed))
    f32 = torch.float32
    o = dict(hist=hist, hist_n=hist_n, entropy=_zeros(R, dtype=f32), k_star=_zeros(B), h_best=_zeros(B, dtype=f32),
             entropy_ok=_zeros(B, dtype=torch.uint8))
    ws = _scratch(rs.rs_entropy_gate_workspace_size(R, V))
    args = (logits, R, V, _cuda(tree["node_off"]), _cuda(commit), B, p, o["hist"], o["hist_n"], o["entropy"], o["k_star"],
            o["h_best"], o["entropy_ok"], ws)
    return dict(call=rs.rs_entropy_gate, args=args, out=o)


_BUFFER = 4096  # tokens of every request's buffer behind an accept call (only its score table is read)


def _accept_tree(case, seed):
    chain_nodes = case["chains"] * case["chain_len"]
    return _trees(case["B"], case["nodes"] - 1 - chain_nodes, case["chains"], case["chain_len"], case["V"], seed)


def _prepare_accept(case, seed):
    B, V, top_c = case["B"], case["V"], case["top_c"]
    tree = _accept_tree(case, seed)
    gen = _generator(seed * 4)
    logits = _logits(tree, V, gen)
    p = rs.params(top_c=top_c, span_len=max(1, case["chain_len"]))
    R = B * tree["N"]
    g = np.random.default_rng([seed, 5])
    sel = np.stack([g.choice(_BUFFER, size=top_c, replace=False) for _ in range(B)]).astype(np.int32)
    sel[:, case["chains"]:] = -1
    f32 = torch.float32
    o = dict(argmax=_zeros(R), topk=_zeros(R, p.beta), lse=_zeros(R, dtype=f32), p_tok=_zeros(R, dtype=f32),
             entropy=_zeros(R, dtype=f32), acc_len=_zeros(B), acc_nodes=_zeros(B, ACC_CAP), bonus=_zeros(B), winner=_zeros(B),
             commit=_zeros(R, dtype=torch.uint8), scores=_scores(B * _BUFFER, gen), status=_zeros(B))
    ws = _scratch(rs.rs_accept_workspace_size(R, V, p.beta))
    args = (logits, R, V, _cuda(tree["node_off"]), B, _cuda(tree["tree_tokens"]), _cuda(tree["parents"]), _cuda(tree["source"]),
            _cuda(tree["chain"]), _cuda(sel), torch.arange(B + 1, device="cuda") * _BUFFER, p, ACC_CAP, o["argmax"], o["topk"], o["lse"],
            o["p_tok"], o["entropy"], o["acc_len"], o["acc_nodes"], o["bonus"], o["winner"], o["commit"], o["scores"], o["status"], ws)
    return dict(call=rs.rs_accept, args=args, out=o)


def _prepare_sample(case, seed):
    B, V = case["B"], case["V"]
    tree = _accept_tree(case, seed)
    gen = _generator(seed * 4)
    logits = _logits(tree, V, gen)
    R = B * tree["N"]
    o = dict(draw=_zeros(R), acc_len=_zeros(B), acc_nodes=_zeros(B, ACC_CAP), bonus=_zeros(B), status=_zeros(B))
    ws = _scratch(rs.rs_tree_sample_workspace_size(R, V))
    args = (logits, R, V, _cuda(tree["node_off"]), B, _cuda(tree["tree_tokens"]), _cuda(tree["parents"]), _cuda(tree["source"]),
            case["temperature"], torch.rand(R, device="cuda", generator=gen), ACC_CAP, o["draw"], o["acc_len"], o["acc_nodes"],
            o["bonus"], o["status"], ws)
    return dict(call=rs.rs_tree_sample, args=args, out=o)


def _retrieval_outputs(B, p):
    return dict(count=_zeros(B), pos=_zeros(B, POS_CAP), sel_pos=_zeros(B, p.top_c), sel_len=_zeros(B, p.top_c),
                spans=_zeros(B, p.top_c, p.span_len), n_sel=_zeros(B), status=_zeros(B))


def _prepare_scan(case, seed):
    B, t = case["B"], case["tokens"]
    X = _tokens(case, seed, B, t)
    p = rs.params(l=max(3, case["k"]), top_c=case["top_c"], span_len=case["span"])
    o = _retrieval_outputs(B, p)
    args = (X, torch.arange(B + 1, device="cuda") * t, B, torch.full((B,), case["k"], dtype=torch.int32, device="cuda"),
            torch.ones(B, dtype=torch.uint8, device="cuda"), _scores(B * t, _generator(seed * 4)), p, POS_CAP, o["count"], o["pos"],
            o["sel_pos"], o["sel_len"], o["spans"], o["n_sel"], o["status"], _scratch(rs.rs_match_scan_workspace_size(B)))
    return dict(call=rs.rs_match_scan, args=args, out=o)


def _prepare_index(case, seed):
    """The token buffers of every step (each request's buffer grows by `append` tokens a step) with the outputs of its query."""
    B, t0, steps, V = case["B"], case["tokens"], case["steps"], case["V"]
    t1 = t0 + steps * case["append"]
    X = _tokens(case, seed, B, t1)
    p = rs.params(l=max(3, case["k"]), top_c=case["top_c"], span_len=case["span"])
    at = lambda n: (X[:, :n].contiguous(), torch.arange(B + 1, device="cuda") * n)  # noqa: E731
    # a serving program reserves room and keeps requests apart; here each step's buffers lie end to end in a tensor of their own
    views = [at(t0 + i * case["append"]) for i in range(steps + 1)]
    return dict(case=case, p=p, views=views, k=torch.full((B,), case["k"], dtype=torch.int32, device="cuda"),
                ok=torch.ones(B, dtype=torch.uint8, device="cuda"), scores=_scores(B * t1, _generator(seed * 4)),
                index=torch.empty(rs.rs_match_index_bytes(B, V, B * t0), dtype=torch.uint8, device="cuda"),
                out=[dict(_retrieval_outputs(B, p), append_status=_zeros(B)) for _ in range(steps)])


def _prepare_step(case, seed):
    B, V, Hq, Hkv, D = case["B"], case["V"], case["Hq"], case["Hkv"], case["D"]
    p = rs.params(top_c=case["top_c"], span_len=max(1, case["chain_len"]))
    x = _attn_inputs(case, seed)
    tree = x["tree"]
    gen = _generator(seed * 4 + 2)
    lens = x["ctx"].astype(np.int64) + 1
    tok_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    X = _tokens(case, seed, B, int(lens.max())).cpu().numpy()
    g = np.random.default_rng([seed, 5])
    sel = np.full((B, p.top_c), -1, np.int32)
    for b in range(B):
        sel[b, : case["chains"]] = g.choice(int(lens[b]) - 1, size=case["chains"], replace=False)
    commit = (g.random(x["R"]) < 0.1).astype(np.uint8)
    commit[:: tree["N"]] = 1
    hist, hist_n = _history(B, p.l, seed)
    bits = lambda a: a.view(torch.int16).cpu().numpy().view(np.uint16)  # noqa: E731
    arrays = dict(logits=_logits(tree, V, gen).cpu().numpy(), node_off=tree["node_off"], row_commit=commit, hist=hist, hist_n=hist_n,
                  tokens=np.concatenate([X[b, : lens[b]] for b in range(B)]), tok_off=tok_off,
                  scores=_scores(B * (case["ctx_hi"] + 1), gen).cpu().numpy(), q=bits(x["q"]), k=bits(x["k"]), v=bits(x["v"]),
                  kv_off=x["kv_off"], ctx_len=x["ctx"], parents=tree["parents"], tree_tokens=tree["tree_tokens"], source=tree["source"],
                  chain=tree["chain"], sel_pos=sel)
    st = VerifyStep(arrays, p, Hq, Hkv, D, pos_cap=POS_CAP, acc_cap=ACC_CAP)
    state = dict(step=st, graph=None, out=dict(st.out, hist=st.d["hist"], hist_n=st.d["hist_n"], scores=st.d["scores"]))
    if case["graph"]:  # the steady state: row entropies come from the previous step's rs_accept
        st.prime()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            st.step()
        torch.cuda.current_stream().wait_stream(side)
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            st.step()
        st.reset_state()
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    if "call" in state:
        state["call"](*state["args"])
        return state["out"]
    if "step" in state:
        if state["graph"] is not None:
            state["graph"].replay()
        else:
            state["step"].step(fused=False)
        return state["out"]
    case, p, index = state["case"], state["p"], state["index"]
    B, V, total = case["B"], case["V"], case["B"] * case["tokens"]
    X, off = state["views"][0]
    rs.rs_match_index_build(X, off, B, V, total, index)
    for (X, off), o in zip(state["views"][1:], state["out"]):
        rs.rs_match_index_append(X, off, B, V, total, index, o["append_status"])
        rs.rs_match_scan_indexed(X, off, B, state["k"], state["ok"], state["scores"], p, POS_CAP, o["count"], o["pos"], o["sel_pos"],
                                 o["sel_len"], o["spans"], o["n_sel"], o["status"], V, total, index)
    return state["out"]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    path, B = case["path"], case["B"]
    nbytes = flops = 0.0
    if path in ("attn", "step"):
        N = 1 + case["model"] + case["chains"] * case["chain_len"]
        Hq, Hkv, D = case["Hq"], case["Hkv"], case["D"]
        keys = B * ((case["ctx_lo"] + case["ctx_hi"]) / 2 + N)
        nbytes += keys * Hkv * D * 4 + B * N * Hq * (D * 6 + 4)
        flops += 4.0 * N * keys * Hq * D
        if path == "step":
            nbytes += B * N * case["V"] * 4 + B * (case["ctx_lo"] + case["ctx_hi"]) / 2 * 4
            flops += 4.0 * B * N * case["V"]
    elif path in ("gate", "accept", "sample"):
        rows = B * case["nodes"]
        nbytes += rows * case["V"] * 4 + rows * 32
        flops += 4.0 * rows * case["V"]
    elif path == "scan":
        nbytes += B * (case["tokens"] * 4 + POS_CAP * 4)
    else:
        nbytes += B * (case["tokens"] * 8 + case["steps"] * POS_CAP * 4)  # each token read, each position written to its list
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """Retrieval and sampling return whole numbers, the same in every implementation."""
    path = case["path"]
    if path in ("attn", "step"):
        # P is rounded to bf16 (2^-9 relative each, averaged over the keys): 0.0017 from the 64-bit result
        return dict(rel=6e-3, max=0.05)
    if path in ("gate", "accept"):
        return dict(rel=1e-5, max=1e-4)  # fp32 sums and exponentials over a row; p_tok, an exponential of a difference, is 2.6e-6 off
    return "exact"


# ------------------------------------------------------------------ the same in 64 bits
def _exact_attn(x, case):
    G, D, scale = case["Hq"] // case["Hkv"], case["D"], case["D"] ** -0.5
    N = x["tree"]["N"]
    out = torch.empty(x["R"], case["Hq"], D, dtype=torch.float64, device="cuda")
    lse = torch.empty(x["R"], case["Hq"], dtype=torch.float64, device="cuda")
    for b in range(case["B"]):
        par = x["tree"]["parents"][b * N:(b + 1) * N]
        see = np.zeros((N, N), bool)
        for i in range(N):
            a = i
            while a >= 0:
                see[i, a] = True
                a = par[a]
        S, k0 = int(x["ctx"][b]), int(x["kv_off"][b])
        mask = torch.cat([torch.ones(N, S, dtype=torch.bool, device="cuda"), _cuda(see)], dim=1).repeat_interleave(G, dim=0)
        rows = slice(b * N, (b + 1) * N)
        for h in range(case["Hkv"]):
            K, V = (x[n][k0:k0 + S + N, h].double() for n in ("k", "v"))
            q = x["q"][rows, h * G:(h + 1) * G].double().reshape(N * G, D)
            s = (q @ K.T * scale).masked_fill_(~mask, -math.inf)
            m = torch.logsumexp(s, dim=1)
            out[rows, h * G:(h + 1) * G] = (torch.exp(s - m[:, None]) @ V).view(N, G, D)
            lse[rows, h * G:(h + 1) * G] = m.view(N, G)
    return out, lse


def _exact_rows(z):
    """Log-sum-exp and entropy (nats) of every row."""
    lse, ent = torch.empty(len(z), dtype=torch.float64, device="cuda"), torch.empty(len(z), dtype=torch.float64, device="cuda")
    for r in range(0, len(z), 64):
        d = z[r:r + 64].double()
        lse[r:r + 64] = torch.logsumexp(d, dim=1)
        ent[r:r + 64] = lse[r:r + 64] - (torch.exp(d - lse[r:r + 64, None]) * d).sum(dim=1)
    return lse, ent


def _exact_p_tok(z, lse, tree):
    parents, tokens = torch.from_numpy(tree["parents"]).cuda().long(), torch.from_numpy(tree["tree_tokens"]).cuda().long()
    rows = torch.arange(len(z), device="cuda")
    up = (rows // tree["N"]) * tree["N"] + parents.clamp(min=0)
    return torch.where(parents < 0, 1.0, torch.exp(z[up, tokens].double() - lse[up]))


def exact(case, seed):
    path = case["path"]
    if path == "attn":
        x = _attn_inputs(case, seed)
        out, lse = _exact_attn(x, case)
        return dict(out=out, lse=lse, status=None)
    if path == "gate":
        tree = _trees(case["B"], case["nodes"] - 1, 0, 0, case["V"], seed)
        _, ent = _exact_rows(_logits(tree, case["V"], _generator(seed * 4)))
        return dict(entropy=ent)
    if path == "accept":
        tree = _accept_tree(case, seed)
        z = _logits(tree, case["V"], _generator(seed * 4))
        lse, ent = _exact_rows(z)
        return dict(lse=lse, entropy=ent, p_tok=_exact_p_tok(z, lse, tree))
    if path == "step":
        x = _attn_inputs(case, seed)
        out, attn_lse = _exact_attn(x, case)
        tree = x["tree"]
        z = _logits(tree, case["V"], _generator(seed * 4 + 2))
        lse, ent = _exact_rows(z)
        o = dict(attn_out=out, attn_lse=attn_lse, lse=lse, acc_entropy=ent, p_tok=_exact_p_tok(z, lse, tree))
        return o if case["graph"] else dict(o, entropy=ent)
    return None
