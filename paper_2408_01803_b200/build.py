"""Builds the CUDA library (libstb.so) for sm_100a with nvcc, and the native host path of its Python calls (_stb_bind.so)
with g++ against the installed torch, in-tree."""
from __future__ import annotations

import os
import re
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libstb.so")
BIND = os.path.join(HERE, "_stb_bind.so")
BIND_FOR = os.path.join(OBJ, "stb_bind.for")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
         "-Xcompiler", "-fPIC"]


def nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return exe


def sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers_mtime() -> float:
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    hs.append(os.path.join(HERE, "..", "include", "stb.h"))
    return max(os.path.getmtime(h) for h in hs)


def _torch_dir() -> str:
    """Where torch is installed (found without importing it)."""
    from importlib.util import find_spec
    return os.path.dirname(find_spec("torch").origin)


def _bind_target(torch_dir: str) -> str:
    """What _stb_bind.so is built for: the installed torch and this interpreter's extension ABI."""
    with open(os.path.join(torch_dir, "version.py")) as f:
        version = re.search(r"__version__\s*=\s*['\"]([^'\"]+)", f.read()).group(1)
    return "torch %s %s" % (version, sysconfig.get_config_var("EXT_SUFFIX"))


def build_bind(force: bool = False) -> str:
    """Compile csrc/stb_bind.cpp into _stb_bind.so, unless the one there is newer than its sources and for the same torch."""
    src = os.path.join(CSRC, "stb_bind.cpp")
    newest = max(os.path.getmtime(src), os.path.getmtime(os.path.join(HERE, "..", "include", "stb.h")))
    torch_dir = _torch_dir()
    target = _bind_target(torch_dir)
    built_for = ""
    if os.path.exists(BIND_FOR):
        with open(BIND_FOR) as f:
            built_for = f.read()
    if not force and os.path.exists(BIND) and os.path.getmtime(BIND) >= newest and built_for == target:
        return BIND
    abi = subprocess.run([sys.executable, "-c", "import torch; print(int(torch._C._GLIBCXX_USE_CXX11_ABI))"], capture_output=True, text=True, check=True)
    inc, lib = os.path.join(torch_dir, "include"), os.path.join(torch_dir, "lib")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    tmp = BIND + ".tmp%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", tmp, src, "-I" + sysconfig.get_paths()["include"], "-I" + inc,
           "-I" + os.path.join(inc, "torch", "csrc", "api", "include"), "-I" + cuda, "-D_GLIBCXX_USE_CXX11_ABI=" + abi.stdout.split()[-1],
           "-L" + lib, "-Wl,-rpath," + lib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("g++ failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
    os.replace(tmp, BIND)
    os.makedirs(OBJ, exist_ok=True)
    with open(BIND_FOR, "w") as f:
        f.write(target)
    return BIND


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every csrc/*.cu for sm_100a (one nvcc per file, in parallel), link libstb.so, and build _stb_bind.so."""
    os.makedirs(OBJ, exist_ok=True)
    hm = _headers_mtime()
    todo, objs = [], []
    for f in sources():
        src, obj = os.path.join(CSRC, f), os.path.join(OBJ, f[:-3] + ".o")
        objs.append(obj)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hm):
            todo.append((src, obj))

    def compile_one(job):
        src, obj = job
        cmd = [nvcc()] + FLAGS + (["-Xptxas=-v"] if verbose else []) + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
        return r.stderr

    pool = ThreadPoolExecutor(max_workers=1)
    bind = pool.submit(build_bind, force)
    if todo:
        with ThreadPoolExecutor(max_workers=min(8, len(todo))) as ex:
            for log in ex.map(compile_one, todo):
                if verbose and log:
                    print(log)
    if todo or not os.path.exists(LIB):
        tmp = LIB + ".tmp%d" % os.getpid()
        subprocess.check_call([nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp] + objs + ["-lcuda"])
        os.replace(tmp, LIB)
    bind.result()
    pool.shutdown()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
