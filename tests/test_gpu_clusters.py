"""Retrieval in a context that can run no cluster of 16 CTAs: the calls of few
requests take clusters of 8 and give the same answers (every retrieval test again
in a process whose library is told so, as the answer is kept with the context)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_clusters_of_eight_for_few_requests():
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider",
                        os.path.join(HERE, "test_gpu_retrieval_sizes.py")],
                       env=dict(os.environ, RS_DEBUG_MATCH_CLUSTER="8"), cwd=os.path.dirname(HERE), capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]


CAPTURED = """
import torch
from paper_2511_01282_gb300 import respec as rs
tok = torch.tensor([9, 7, 1, 2, 7, 3, 4, 7], dtype=torch.int32, device="cuda")
off, k, sc = torch.tensor([0, 8], device="cuda"), torch.ones(1, dtype=torch.int32, device="cuda"), torch.full((8,), 0.5, device="cuda")
out = [torch.full((n,), -7, dtype=torch.int32, device="cuda") for n in (1, 4, 3, 3, 24, 1, 1)]
idx = torch.empty(rs.rs_match_index_bytes(1, 16, 8), dtype=torch.uint8, device="cuda")
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    rs.rs_match_scan(tok, off, 1, k, None, sc, rs.params(), 4, *out)
    rs.rs_match_index_build(tok, off, 1, 16, 8, idx)
h = torch.cuda.CUDAGraph()
with torch.cuda.graph(h):
    rs.rs_match_scan_indexed(tok, off, 1, k, None, sc, rs.params(), 4, *out, 16, 8, idx)
for graph in (g, h):
    for o in out:
        o.fill_(-7)
    graph.replay()
    torch.cuda.synchronize()
    assert out[0].tolist() == [2] and out[1].tolist() == [1, 4, -1, -1] and out[6].tolist() == [0], [o.tolist() for o in out]
"""


def test_the_first_call_of_a_process_may_be_captured():
    r = subprocess.run([sys.executable, "-c", CAPTURED], cwd=os.path.dirname(HERE), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
