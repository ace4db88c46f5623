"""Builds the CUDA shared library in-tree with nvcc for sm_100a.

    python -m paper_2407_19947_b200.build [--force]
"""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess
import sys
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_PATH = os.path.join(HERE, "libstairs_b200.so")
# variants of the whole-pass kernel (head size, model family, attention path, at most 16 rows, shared rows), one object each
FORWARD = [v + (s,) for s in (0, 1) for v in ([(64, 1, a, o) for a in (0, 1) for o in (0, 1)] + [(64, 2, a, o) for a in (0, 1) for o in (0, 1)] +
           [(80, 2, 0, o) for o in (0, 1)] + [(128, 2, a, o) for a in (0, 1) for o in (0, 1)] + [(0, 0, 3, 0)])]
NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-Xptxas", "-v"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libstairs_b200.so")


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "stairs.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles csrc/*.cu into libstairs_b200.so (skipped when up to date).  Returns the path."""
    if not force and not _stale():
        return LIB_PATH
    jobs = [("engine.cu", [])] + [("forward.cu", ["-DFWD_HD=%d" % hd, "-DFWD_FAM=%d" % fam, "-DFWD_ATT=%d" % att, "-DFWD_ONE=%d" % one, "-DFWD_SHARE=%d" % share])
                                  for hd, fam, att, one, share in FORWARD]
    log = ""
    failed = False
    with tempfile.TemporaryDirectory() as tmp:
        cmds = [[_nvcc()] + NVCC_FLAGS + defs + ["-c", "-o", os.path.join(tmp, "%d.o" % i), os.path.join(CSRC, src)]
                for i, (src, defs) in enumerate(jobs)]
        with concurrent.futures.ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as pool:
            results = list(pool.map(lambda c: subprocess.run(c, capture_output=True, text=True), cmds))
        cmds.append([_nvcc(), "-shared", "-Xlinker", "-z", "-Xlinker", "defs", "-o", LIB_PATH] + [os.path.join(tmp, "%d.o" % i) for i in range(len(jobs))])
        if all(r.returncode == 0 for r in results):
            results.append(subprocess.run(cmds[-1], capture_output=True, text=True))
        for cmd, r in zip(cmds, results):
            log += " ".join(cmd) + "\n" + r.stdout + r.stderr
            failed = failed or r.returncode != 0
    with open(os.path.join(HERE, "build.log"), "w") as f:
        f.write(log)
    if failed:
        raise RuntimeError("nvcc failed:\n" + log[-6000:])
    if verbose:
        print(log)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
