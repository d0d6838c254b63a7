"""Build the CUDA library in-tree with nvcc for sm_100a, and the extension module of the calls (g++)."""
from __future__ import annotations

import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgsi_b200.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


HASH = LIB + ".srchash"


def _source_hash() -> str:
    import hashlib
    h = hashlib.sha256()
    deps = sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + \
        sorted(glob.glob(os.path.join(ROOT, "include", "*.h")))
    for p in deps:
        h.update(os.path.basename(p).encode())
        h.update(open(p, "rb").read())
    h.update(" ".join(NVCC_FLAGS).encode())
    return h.hexdigest()


def _stale() -> bool:
    """The library is current iff it was built from exactly these sources
    (content hash; file times do not survive a copy to another machine)."""
    if not os.path.exists(LIB) or not os.path.exists(HASH):
        return True
    return open(HASH).read().strip() != _source_hash()


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libgsi_b200.so (cross-compiles without a GPU).  The translation
    units are compiled side by side (one nvcc process each), then linked."""
    if not force and not _stale():
        return LIB
    import shutil
    import tempfile
    from concurrent.futures import ThreadPoolExecutor
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    compile_flags = [f for f in NVCC_FLAGS if f != "-shared"]
    inc = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    objdir = tempfile.mkdtemp(prefix="gsi_build_")

    def compile_one(src: str) -> str:
        obj = os.path.join(objdir, os.path.basename(src) + ".o")
        cmd = [nvcc, *compile_flags, *inc, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            print(r.stdout + r.stderr, flush=True)
        if r.returncode != 0:
            raise subprocess.CalledProcessError(r.returncode, cmd)
        return obj

    try:
        with ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as pool:
            objs = list(pool.map(compile_one, sources()))
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.check_call([nvcc, *NVCC_FLAGS, "-o", tmp, *objs])
        os.replace(tmp, LIB)
    finally:
        shutil.rmtree(objdir, ignore_errors=True)
    with open(HASH, "w") as f:
        f.write(_source_hash())
    return LIB


# The extension module of the calls (torch_calls.cpp): beside the library, built for this torch and Python.
CALLS_SRC = os.path.join(CSRC, "torch_calls.cpp")
CALLS = os.path.join(HERE, "_torch_calls.so")


def _calls_flags() -> list[str]:
    import torch
    return ["-O2", "-std=c++17", "-fPIC", "-shared", "-DTORCH_EXTENSION_NAME=_torch_calls",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]


def _calls_command(out: str) -> list[str]:
    import sysconfig
    import torch
    base = os.path.join(os.path.dirname(torch.__file__))
    inc = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], "/usr/local/cuda/include", os.path.join(ROOT, "include")]
    return ["g++", *[f"-I{d}" for d in inc], CALLS_SRC, "-o", out, "-L" + os.path.join(base, "lib"), *_calls_flags()]


def _calls_hash() -> str:
    """What the module was built from and for: the sources, the flags, this torch and this Python's binary
    interface.  No path: the module is built once and used where the tree is copied to."""
    import hashlib
    import sysconfig
    import torch
    h = hashlib.sha256(" ".join([*_calls_flags(), torch.__version__, sysconfig.get_config_var("SOABI")]).encode())
    for p in (CALLS_SRC, os.path.join(ROOT, "include", "gsi.h")):
        h.update(open(p, "rb").read())
    return h.hexdigest()


def build_calls(force: bool = False) -> str:
    digest, stamp = _calls_hash(), CALLS + ".srchash"
    if not force and os.path.exists(CALLS) and os.path.exists(stamp) and open(stamp).read().strip() == digest:
        return CALLS
    tmp = CALLS + f".tmp{os.getpid()}"
    subprocess.check_call(_calls_command(tmp))
    os.replace(tmp, CALLS)
    with open(stamp, "w") as f:
        f.write(digest)
    return CALLS


if __name__ == "__main__":
    import sys
    build_calls("--force" in sys.argv)
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
