"""In-tree build of the CUDA library: nvcc -> paper_2407_08454_b200/libkvm.so (sm_100a only)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB = os.path.join(_PKG, "libkvm.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--expt-relaxed-constexpr", "--expt-extended-lambda", "-Xcompiler", "-fPIC",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


# A second library for the tests of the give-up paths of the bounded device waits: the same sources with a short
# wait limit and producers that leave out one stage (the prefill attention's in every block, the score passes' and the decode attention's in one),
# so that a wait runs out, the kernel returns and reports it.  It is never loaded by the package itself.
WAITTEST_LIB = os.path.join(_PKG, "libkvm_waittest.so")
WAITTEST_FLAGS = ("-DKVM_TEST_WAIT_LIMIT_CLOCKS=4000000ll", "-DKVM_TEST_DROP_B_STAGE=3", "-DKVM_TEST_DROP_SCORE_STEP=0",
                  "-DKVM_TEST_DROP_ATTEND_STAGE=0", "-DKVM_TEST_DROP_CTA=1")


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(_ROOT, "include", "*.h"))
    return any(os.path.getmtime(f) > t for f in deps)


def build(force: bool = False, verbose: bool = False, extra=(), lib: str = LIB) -> str:
    """Compile every .cu under csrc/ into one shared library.  Returns its path."""
    if not force and not _stale(lib):
        return lib
    nvcc = os.environ.get("NVCC", "nvcc")
    objdir = os.path.join(_PKG, "_build" + os.path.basename(lib)[len("libkvm"):-len(".so")])
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, *extra, "-I", os.path.join(_ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip() and (verbose or p.returncode != 0):
            print(out, file=sys.stderr)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = lib + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs,
                           "-lcudart_static", "-ldl", "-lrt", "-lpthread"])
    os.replace(tmp, lib)
    return lib


def build_waittest(force: bool = False) -> str:
    """The test-only library with a short wait limit and a dropped producer stage (see WAITTEST_FLAGS)."""
    return build(force=force, extra=WAITTEST_FLAGS, lib=WAITTEST_LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True,
                extra=("-Xptxas", "-v") if "--ptxas" in sys.argv else ()))
