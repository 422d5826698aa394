"""In-tree build of libstateflow.so for sm_100a (nvcc cross-compiles without a GPU)."""
from __future__ import annotations

import glob
import os
import subprocess
import tempfile

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libstateflow.so")

SOURCES = ["stateflow.cu", "variants.cu", "delta_chunked.cu", "channel_chunked.cu"]

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    srcs = glob.glob(os.path.join(CSRC, "*")) + [os.path.join(_HERE, "..", "include", "stateflow.h")]
    return any(os.path.getmtime(s) > t for s in srcs)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + ".tmp%d" % os.getpid()
        # the translation units are compiled side by side, then linked
        with tempfile.TemporaryDirectory() as work:
            objs = [os.path.join(work, f + ".o") for f in SOURCES]
            jobs = [subprocess.Popen([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", "-o", o, os.path.join(CSRC, f)])
                    for f, o in zip(SOURCES, objs)]
            if any([job.wait() != 0 for job in jobs]):
                raise RuntimeError("nvcc failed on %s" % ", ".join(f for f, job in zip(SOURCES, jobs) if job.returncode != 0))
            subprocess.check_call([nvcc] + NVCC_FLAGS + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
