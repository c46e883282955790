"""Build libcredit.so in-tree with nvcc for sm_103a (GB300).

Every translation unit compiles in parallel; the kernel TUs compile once per
input dtype.  The result lands in ``paper_2609_01864_gb300/_build/``.  No
cmake, no torch C++ extension: the library exposes a plain C ABI and is
loaded with ctypes.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OUT = os.path.join(PKG, "_build")
LIB = os.path.join(OUT, "libcredit.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
              f"-I{os.path.join(ROOT, 'include')}", f"-I{CSRC}"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libcredit.so")


def _units():
    units = []
    for tin in (0, 1, 2):
        for name in ("credit_kernels", "credit_team"):
            units.append((os.path.join(CSRC, name + ".cu"), f"{name}_{tin}.o", [f"-DCREDIT_TIN={tin}"]))
        units.append((os.path.join(CSRC, "credit_team.cu"), f"credit_team_traced_{tin}.o",
                      [f"-DCREDIT_TIN={tin}", "-DCREDIT_TRACED=1"]))
    units.append((os.path.join(CSRC, "credit_warps.cu"), "credit_warps_traced.o", ["-DCREDIT_TRACED=1"]))
    for dt in (0, 1):
        units.append((os.path.join(CSRC, "credit_bwd.cu"), f"credit_bwd_{dt}.o", [f"-DCREDIT_BWD_DT={dt}"]))
    for src in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cpp"))):
        if os.path.basename(src) in ("credit_kernels.cu", "credit_team.cu"):
            continue
        units.append((src, os.path.basename(src).rsplit(".", 1)[0] + ".o", []))
    return units


def _deps():
    return (glob.glob(os.path.join(CSRC, "*")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
            + [os.path.abspath(__file__)])


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in _deps())


def build(force: bool = False, verbose: bool = False, jobs: int | None = None) -> str:
    if not force and up_to_date():
        return LIB
    nvcc = _nvcc()
    os.makedirs(OUT, exist_ok=True)
    units = _units()

    def compile_one(u):
        src, obj, extra = u
        cmd = [nvcc, *ARCH, *NVCC_FLAGS, *extra, "-c", src, "-o", os.path.join(OUT, obj)]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)} {extra}:\n{r.stdout}\n{r.stderr}")
        return obj

    jobs = jobs or min(len(units), max(2, os.cpu_count() or 2))
    with cf.ThreadPoolExecutor(jobs) as ex:
        objs = list(ex.map(compile_one, units))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *[os.path.join(OUT, o) for o in objs], "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
