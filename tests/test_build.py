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


def test_another_torch_rebuilds_the_binding(monkeypatch, tmp_path):
    # files of an older torch that is installed later are older than the binding
    made = []
    real = subprocess.run
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: made.append(cmd) or real(["true"], **kw))
    monkeypatch.setattr(build.os, "replace", lambda a, b: None)
    monkeypatch.setattr(build, "_write", lambda path, text: None)
    build.build()
    assert not made                                   # nothing to do
    other = tmp_path / "torch"
    (other / "include").mkdir(parents=True)
    (other / "version.py").write_text("__version__ = '2.0.0'\n")
    os.utime(other / "version.py", (0, 0))
    monkeypatch.setattr(build, "_torch_dir", lambda: str(other))
    build.build()
    assert any(build.BIND_SRC in c for c in made) and any(str(other / "include") in c for c in made)
    assert any("-shared" in c and any(a.startswith(build.BIND) for a in c) for c in made)
    assert not any(c[0].endswith("nvcc") for c in made)


def test_the_library_builds_without_torch(monkeypatch):
    monkeypatch.setattr(build.importlib.util, "find_spec", lambda name: None)
    assert build.build() == build.LIB and os.path.exists(build.LIB)
