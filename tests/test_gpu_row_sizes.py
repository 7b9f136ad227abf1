"""Draws at the ends of rows whose last chunk of 8192 logits holds a few only,
for rows read by eight, four and single logits, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import test_gpu_sample

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("V", [1, 31, 8184, 8191, 8192, 8193, 8196, 8200, 8223, 8225, 16385, 40001, 40004, 40008])
@pytest.mark.parametrize("lead", [0, 1])
def test_draws_at_the_ends_of_rows(V, lead, monkeypatch):
    # lead: rows that begin one logit past a 16-byte boundary, whatever V
    def to_cuda(a, cuda=test_gpu_sample._cuda):
        if a.ndim != 2:
            return cuda(a)
        flat = torch.zeros(a.size + lead, device="cuda")
        flat[lead:] = cuda(a).reshape(-1)
        return flat[lead:].view(a.shape)

    monkeypatch.setattr(test_gpu_sample, "_cuda", to_cuda)
    rng = np.random.default_rng(V + lead)
    R = 6
    logits = rng.standard_normal((R, V)).astype(np.float32)
    logits[1, :-1] -= 60.0                    # nearly all the mass on the last id
    logits[2, :max(V - 40, 0)] = -np.inf      # all of it on the last forty
    logits[3, max(V - 3, 1):] = -np.inf       # none on the last ones
    logits[4, 1:] -= 60.0                     # on the first
    node_off = np.array([0, R], np.int32)
    parents = np.array([-1, 0, 1, 2, 3, 4], np.int32)
    tokens = rng.integers(0, V, R).astype(np.int32)
    source = np.ones(R, np.uint8)
    for u in (0.0, 0.37, 0.999, np.nextafter(np.float32(1), np.float32(0))):
        test_gpu_sample.check(logits, node_off, tokens, parents, source, 1.0, np.full(R, u))
