"""Row statistics of rows with infinite logits and masks, for rows of one chunk, of
a cluster and of more chunks than a warp has lanes."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import host
from paper_2511_01282_gb300 import respec as rs
from test_gpu_index import _cuda

pytestmark = pytest.mark.gpu
SIZES = [1024, 8192, 20000, 70001, 280000]  # 280000: 35 chunks of 8192


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def gate_entropy(z):
    R, V = z.shape
    p = rs.params()
    z0 = lambda *s, dtype=torch.int32: torch.zeros(s, dtype=dtype, device="cuda")  # noqa: E731
    f32 = torch.float32
    ent = z0(R, dtype=f32)
    ws = torch.empty(max(256, rs.rs_entropy_gate_workspace_size(R, V)), dtype=torch.uint8, device="cuda")
    rs.rs_entropy_gate(_cuda(z), R, V, _cuda(np.array([0, R], np.int32)), z0(R, dtype=torch.uint8), 1, p, z0(1, p.l, dtype=f32), z0(1),
                       ent, z0(1), z0(1, dtype=f32), z0(1, dtype=torch.uint8), ws)
    return host(ent).astype(np.float64)


def accept_rows(z, with_entropy=True):
    """Row statistics of rs_accept over a tree of one path, and its p_tok (each node's token is its parent's best)."""
    R, V = z.shape
    p = rs.params(top_c=1)
    par = np.arange(-1, R - 1, dtype=np.int32)
    tok = np.concatenate([[0], z[:-1].argmax(1)]).astype(np.int32)
    src, chn = np.concatenate([[0], np.ones(R - 1)]).astype(np.uint8), np.full(R, -1, np.int8)
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")  # noqa: E731
    flt = lambda n: torch.zeros(n, device="cuda")                         # noqa: E731
    o = dict(argmax=i32(R), topk=i32(R, p.beta), lse=flt(R), p_tok=flt(R), entropy=flt(R), acc_len=i32(1), acc_nodes=i32(1, 8),
             bonus=i32(1), winner=i32(1), commit=torch.zeros(R, dtype=torch.uint8, device="cuda"), scores=flt(8), status=i32(1))
    ws = torch.empty(rs.rs_accept_workspace_size(R, V, p.beta), dtype=torch.uint8, device="cuda")
    rs.rs_accept(_cuda(z), R, V, _cuda(np.array([0, R], np.int32)), 1, _cuda(tok), _cuda(par), _cuda(src), _cuda(chn), i32(1, 1),
                 _cuda(np.array([0, 8], np.int64)), p, 8, o["argmax"], o["topk"], o["lse"], o["p_tok"],
                 o["entropy"] if with_entropy else None, o["acc_len"], o["acc_nodes"], o["bonus"], o["winner"], o["commit"],
                 o["scores"], o["status"], ws)
    return {k: host(v) for k, v in o.items()}


@pytest.mark.parametrize("V", SIZES)
def test_a_slice_without_mass_counts_for_nothing(V):
    # a +inf logit takes the mass of the logits that its warp sums (every eighth run
    # of `lanes` ids of a chunk), and no more
    rng = np.random.default_rng(V)
    z = rng.standard_normal((3, V)).astype(np.float32)
    z[0, 5] = z[1, V - 1] = z[2, V // 2] = np.inf
    for got, lanes in ((gate_entropy(z), 256 if V % 8 == 0 else 128 if V % 4 == 0 else 32),
                       (accept_rows(z)["entropy"].astype(np.float64), 128 if V % 4 == 0 else 32)):
        rest = z.astype(np.float64)
        ids = np.arange(V)
        for r in range(3):
            at = int(np.argmax(z[r]))
            rest[r, (ids // 8192 == at // 8192) & (ids % 8192 // lanes % 8 == at % 8192 // lanes % 8)] = -np.inf
        assert np.abs(got - oracle.entropy_rows(rest.astype(np.float32))).max() < 1e-3


@pytest.mark.parametrize("V", SIZES)
@pytest.mark.parametrize("mask", [-np.finfo(np.float32).max, -2.5e38, -1e30, -1e10, -1e9, -4e8, -65504])
def test_masks_of_the_lowest_value(V, mask):
    # masked ids in whole chunks, in whole slices of a warp, alone, and everywhere
    # but at one id: they carry no mass, whatever the finite value
    rng = np.random.default_rng(V)
    z = (3 * rng.standard_normal((7, V))).astype(np.float32)
    ids = np.arange(V)
    z[0, max(1, V // 3):] = mask
    z[1, :V - 5] = mask
    z[2, ids // 128 % 8 != 3] = mask
    z[3, ids % 3 != 1] = mask
    z[4, ids != V // 2] = mask
    z[5, :] = mask                       # nothing is left: a uniform row
    z[6, ids % 2 == 0] = -np.inf
    H = oracle.entropy_rows(z)
    assert np.abs(gate_entropy(z) - H).max() < 1e-3
    zd = z.astype(np.float64)
    m = zd.max(1)
    lse = m + np.log(np.exp(zd - m[:, None]).sum(1))
    for with_entropy in (True, False):
        o = accept_rows(z, with_entropy)
        if with_entropy:
            assert np.abs(o["entropy"].astype(np.float64) - H).max() < 1e-3
        assert np.allclose(o["lse"].astype(np.float64), lse, rtol=1e-5, atol=1e-6)
        p = np.exp(m[:-1] - lse[:-1])    # every node's token is its parent's best
        got = o["p_tok"][1:].astype(np.float64)
        assert np.allclose(np.delete(got, 5), np.delete(p, 5), rtol=1e-4, atol=1e-7)
        assert 0 <= got[5] <= 1          # both logit and lse are the mask: ln V may be below its rounding
        assert (o["argmax"] == z.argmax(1)).all()
