"""The in-tree build: what it takes for out of date, and which library the binding
ends up with."""
import os
import subprocess
import sys

import pytest

from paper_2511_01282_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def test_the_binding_calls_the_library_beside_it(tmp_path):
    # another librespec.so on the loader's path (an older installation, say) is not taken for it
    decoy = tmp_path / "decoy.c"
    decoy.write_text("int rs_match_scan(void) { return 4; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", str(decoy), "-o", str(tmp_path / "librespec.so")], check=True)
    code = ("from paper_2511_01282_gb300 import respec as rs\n"
            "rs.rs_match_scan(16, 16, 0, 16, None, 16, rs.params(), 4, *([16] * 7), None, stream=0)\n")
    path = str(tmp_path) + os.pathsep + os.environ.get("LD_LIBRARY_PATH", "")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, LD_LIBRARY_PATH=path), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-1500:]
