"""Build the lMBD CUDA library in-tree (sm_103a), no CMake.

``python -m paper_2407_06409_gb300.build`` or ``build()`` compiles every ``.cu``
file of ``csrc/`` in parallel with nvcc and links ``_lib/liblmbd.so``.  An object is
kept when its source, the headers, the compiler and the flags are those it was made
from (a digest beside it), so that every test module can call ``build()``.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import hashlib
import os
import platform
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_lib")
LIB = os.path.join(OUT, "liblmbd.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def sources() -> list[str]:
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _digest(cmd: list[str], files: list[str]) -> str:
    """Of a command and all it reads, on this machine's architecture."""
    h = hashlib.sha256()
    nvcc = os.stat(os.path.realpath(cmd[0]))
    h.update(repr((platform.machine(), nvcc.st_size, nvcc.st_mtime_ns, cmd)).encode())
    for f in files:
        with open(f, "rb") as fh:
            data = fh.read()
        h.update(f"{os.path.basename(f)} {len(data)} ".encode() + data)
    return h.hexdigest()


def _up_to_date(target: str, digest: str) -> bool:
    """Was target made from this?  If not, its digest goes, so that a build cut short leaves none."""
    path = target + ".digest"
    if not os.path.exists(path):
        return False
    with open(path) as fh:
        if os.path.exists(target) and fh.read() == digest:
            return True
    os.remove(path)
    return False


def _made(target: str, digest: str) -> None:
    with open(target + ".digest", "w") as fh:
        fh.write(digest)


def build(verbose: bool = False, extra: list[str] | None = None) -> str:
    """Compile and link; returns the path of the shared library."""
    os.makedirs(OUT, exist_ok=True)
    nvcc = _nvcc()
    srcs = sources()
    objs = [os.path.join(OUT, os.path.basename(s)[:-3] + ".o") for s in srcs]
    extra = list(extra or [])
    headers = sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(HERE, "..", "include", "*.h")))

    def comp(pair):
        src, obj = pair
        cmd = [nvcc, *ARCH, *FLAGS, *extra, "-c", src, "-o", obj]
        digest = _digest(cmd, [src, *headers])
        if _up_to_date(obj, digest) and not verbose:
            return cmd, None, digest
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode == 0:
            _made(obj, digest)
        return cmd, r, digest

    digests = []
    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        for cmd, r, digest in ex.map(comp, zip(srcs, objs)):
            digests.append(digest)
            if r and (verbose or r.returncode):
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
            if r and r.returncode:
                raise RuntimeError("nvcc failed for " + cmd[-3])
    cmd = [nvcc, *ARCH, "-shared", "-o", LIB + ".tmp", *objs, "-lcudart"]
    digest = _digest(cmd + digests, [])
    if _up_to_date(LIB, digest):
        return LIB
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        raise RuntimeError("link failed")
    os.replace(LIB + ".tmp", LIB)
    _made(LIB, digest)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv))
