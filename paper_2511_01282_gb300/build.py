"""Build ``librespec.so`` (sm_103a) and its Python binding in-tree.

Each CUDA translation unit under ``csrc/`` is compiled in parallel with nvcc,
then linked into one shared library next to this file.  The CUDA runtime is
linked statically, so the library needs only the driver at run time.
``csrc/bind.cpp`` (the marshalling of ``respec.py``) is compiled beside them
with g++ against the installed torch; it gets the library's entry points from
``respec.py``, which loads the library by its path.  Without torch only the
library is built (for callers of the C ABI).
"""
import concurrent.futures as cf
import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "librespec.so")
BIND_SRC = os.path.join(CSRC, "bind.cpp")
BIND = os.path.join(HERE, "_respec_bind.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc():
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _torch_dir():
    spec = importlib.util.find_spec("torch")
    return None if spec is None else list(spec.submodule_search_locations)[0]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    return hs + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE) if f.endswith(".h")]


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _read(path):
    if not os.path.exists(path):
        return None
    with open(path) as f:
        return f.read()


def _write(path, text):
    with open(path, "w") as f:
        f.write(text)


def build(force=False, verbose=False, extra_flags=()):
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)
    hdrs = _headers()
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE,
                    "-I", CSRC, "--expt-relaxed-constexpr"] + list(extra_flags)
    jobs = []
    objs = []
    for src in sources():
        obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + hdrs):
            jobs.append([nvcc] + flags + ["-c", src, "-o", obj])

    torch_dir = _torch_dir()
    cuda_include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    bind_obj = os.path.join(BUILD, "bind.o")
    # the torch that the binding is for, by path and version (an older one that is
    # installed later has older files)
    stamp = os.path.join(BUILD, "bind.torch")
    torch_is = torch_dir and torch_dir + "\n" + (_read(os.path.join(torch_dir, "version.py")) or "")
    rebind = torch_dir and (force or _read(stamp) != torch_is or _stale(bind_obj, [BIND_SRC] + hdrs))
    if rebind:
        jobs.append(["g++", "-O2", "-std=c++17", "-fPIC", "-I", INCLUDE, "-I", sysconfig.get_paths()["include"],
                     "-I", os.path.join(torch_dir, "include"),
                     "-I", os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
                     "-I", cuda_include, "-c", BIND_SRC, "-o", bind_obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("compile failed: " + " ".join(cmd))
        return r

    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
            list(ex.map(run, jobs))
    if force or any(j[0] == nvcc for j in jobs) or _stale(LIB, objs + [__file__]):
        tmp = LIB + ".tmp.%d" % os.getpid()
        run([nvcc] + ARCH + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    if torch_dir and (rebind or _stale(BIND, [bind_obj, __file__])):
        tmp = BIND + ".tmp.%d" % os.getpid()
        torch_lib = os.path.join(torch_dir, "lib")
        run(["g++", "-shared", "-o", tmp, bind_obj, "-L", torch_lib, "-ltorch_python", "-ltorch",
             "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath," + torch_lib])
        os.replace(tmp, BIND)
        _write(stamp, torch_is)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
