"""Builds the CUDA library in-tree with nvcc for sm_100a, and the Python extension that marshals its arguments.

The shared objects are written next to this file (libba.so, ba_marshal.so).  Sidecar files
store a hash of the sources and flags so that an up-to-date build is reused.
"""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
import sysconfig
import threading

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(HERE, "libba.so")
STAMP = LIB + ".hash"

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "--expt-relaxed-constexpr",
]


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _digest() -> str:
    h = hashlib.sha256()
    h.update(" ".join(NVCC_FLAGS).encode())
    files = _sources() + sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h")))
    files.append(os.path.join(INCLUDE, "ba.h"))
    for f in files:
        h.update(os.path.basename(f).encode())
        with open(f, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def _compile(cmd, out: str, digest: str, failed: str) -> str:
    """Runs the compiler with `out` as its output, whole: a process that loads `out` meanwhile, or builds it as well, finds the old
    file or the new one.  Returns the compiler's messages."""
    own = f"{out}.{os.getpid()}.{threading.get_ident()}"
    try:
        res = subprocess.run(cmd + ["-o", own], capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(failed + res.stdout + res.stderr)
        os.replace(own, out)
        with open(own, "w") as fh:
            fh.write(digest)
        os.replace(own, out + ".hash")
    finally:
        if os.path.exists(own):
            os.remove(own)
    return res.stderr


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libba.so (if needed) and return its path."""
    digest = _digest()
    if not force and os.path.exists(LIB) and os.path.exists(STAMP):
        with open(STAMP) as fh:
            if fh.read().strip() == digest:
                return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc] + NVCC_FLAGS + ["-I", INCLUDE, "-I", CSRC] + _sources()
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
        print(" ".join(cmd), file=sys.stderr)
    messages = _compile(cmd, LIB, digest, "nvcc failed:\n")
    if verbose:
        print(messages, file=sys.stderr)
    return LIB


def build_marshal(force: bool = False) -> str:
    """Compile csrc/ba_marshal.c into ba_marshal.so (if needed) and return its path."""
    out, src, header = os.path.join(HERE, "ba_marshal.so"), os.path.join(CSRC, "ba_marshal.c"), os.path.join(INCLUDE, "ba.h")
    flags = ["-O2", "-fPIC", "-shared", "-Wall", "-Werror"]
    # (what goes into it, not where it lies: a tree that was copied elsewhere keeps its build)
    h = hashlib.sha256(" ".join(flags + [sys.version]).encode())
    for f in (src, header):
        with open(f, "rb") as fh:
            h.update(fh.read())
    digest = h.hexdigest()
    if not force and os.path.exists(out) and os.path.exists(out + ".hash"):
        with open(out + ".hash") as fh:
            if fh.read().strip() == digest:
                return out
    _compile([os.environ.get("CC", "gcc")] + flags + ["-I", sysconfig.get_paths()["include"], "-I", INCLUDE, src], out, digest,
             "the argument marshalling extension failed to build:\n")
    return out


if __name__ == "__main__":
    build_marshal(force="--force" in sys.argv)
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
