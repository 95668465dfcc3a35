"""Build step of the CUDA library: nvcc, sm_100a only, in-tree output next to this file."""
from __future__ import annotations

import glob
import os
import subprocess
import tempfile

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libttc_lqr.so")
NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = glob.glob(os.path.join(CSRC, "*")) + glob.glob(os.path.join(_HERE, "..", "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every ``csrc/*.cu`` (side by side) into ``libttc_lqr.so``; rebuilds when a source is newer."""
    if force or _stale():
        nvcc = [os.environ.get("NVCC", "nvcc")] + NVCC_FLAGS
        with tempfile.TemporaryDirectory() as tmp:
            objects, jobs = [], []
            for src in sources():
                objects.append(os.path.join(tmp, os.path.basename(src) + ".o"))
                cmd = nvcc + (["-Xptxas", "-v"] if verbose else []) + ["-c", "-o", objects[-1], src]
                jobs.append((cmd, subprocess.Popen(cmd)))
            failed = [subprocess.CalledProcessError(job.returncode, cmd) for cmd, job in jobs if job.wait()]
            if failed:
                raise failed[0]
            subprocess.run(nvcc + ["-shared", "-o", LIB] + objects, check=True)
    return LIB
