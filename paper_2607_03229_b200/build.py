"""Build libmpipe_enc.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmpipe_enc.so")
HOST_SRC = os.path.join(CSRC, "hostpath.cpp")
HOST_LIB = os.path.join(HERE, "_hostpath.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "--shared", "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + [HOST_SRC] + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        [os.path.join(HERE, "..", "include", "mpipe_enc.h")]


def built_for() -> str:
    """What the marshalling module is compiled against and works with only: torch's and Python's C++ interfaces."""
    import torch
    return f"marshalling for torch {torch.__version__}, {sys.implementation.cache_tag}"


def host_is_current() -> bool:
    """Whether the marshalling module there is was built for this torch and this Python (it carries their names)."""
    with open(HOST_LIB, "rb") as f:
        return built_for().encode() in f.read()


def is_stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(HOST_LIB) or not host_is_current():
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(HOST_LIB))
    return any(os.path.getmtime(f) > t for f in _deps())


def host_command(out: str):
    """The Python marshalling module: plain C++ against Python's and torch's headers."""
    import torch
    tdir = os.path.dirname(torch.__file__)
    inc = [sysconfig.get_paths()["include"], os.path.join(tdir, "include"), os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           "/usr/local/cuda/include"]
    return ([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
             f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DMPIPE_BUILT_FOR="{built_for()}"'] + ["-I" + d for d in inc] +
            [HOST_SRC, "-o", out, "-L" + os.path.join(tdir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"])


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library, and the Python marshalling module.  Returns the library's path."""
    if not force and not is_stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    work = os.path.join(HERE, "build")
    os.makedirs(work, exist_ok=True)
    # both libraries are linked beside the objects, each process under its own name, and moved to their place when everything is there
    tmp, host_tmp = (os.path.join(work, f"{os.getpid()}.{os.path.basename(f)}") for f in (LIB, HOST_LIB))
    try:
        for src in sources():
            obj = os.path.join(work, os.path.basename(src)[:-3] + ".o")
            cmd = [nvcc] + [f for f in NVCC_FLAGS if f != "--shared"] + ["-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
            objs.append(obj)
        procs.append((HOST_SRC, subprocess.Popen(host_command(host_tmp), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        failed = False
        for src, p in procs:
            out, _ = p.communicate()
            if out.strip() and (verbose or p.returncode != 0):
                print(out, file=sys.stderr)
            failed |= p.returncode != 0
        if failed:
            raise RuntimeError("nvcc failed")
        subprocess.run([nvcc] + NVCC_FLAGS + objs + ["-o", tmp], check=True)
        os.replace(host_tmp, HOST_LIB)
        os.replace(tmp, LIB)
    finally:   # (after a failure or an interruption)
        for _, p in procs:
            if p.poll() is None:
                p.kill()
                p.wait()
        for f in (tmp, host_tmp):
            if os.path.exists(f):
                os.remove(f)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
