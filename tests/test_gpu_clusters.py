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
