"""Compile the CUDA library libace_gb300.so for sm_103a, in-tree.

Each .cu under csrc/ becomes one object (compiled in parallel); they are linked with nvcc into
``_build/libace_gb300.so`` next to this file.  Rebuilds only when a source or header is newer
than the library.
"""

from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import re
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libace_gb300.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
LINEINFO = ["-lineinfo"]
NVCC_FLAGS = ["-std=c++17", "-O3", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _units() -> list[tuple[str, str, list[str]]]:
    """(source, object, flags) of every compilation, the long ones first.  line_pair_plane.cu is
    compiled once per axis length of line_pair_shapes.h, without line tables except for one length
    (they would make up 80% of a 200 MB library)."""
    out = []
    with open(os.path.join(CSRC, "line_pair_shapes.h")) as f:
        lengths = [int(x) for x in re.findall(r"X\((\d+)\)", f.read())]
    for src in sources():
        name = os.path.basename(src)[:-3]
        if name == "line_pair_plane":
            out += [(src, f"{name}_{n}.o", [f"-DACE_LP_N2={n}"] + LINEINFO * (n == 96)) for n in lengths]
        else:
            out.append((src, name + ".o", LINEINFO))
    return sorted(out, key=lambda u: "line_pair_plane" not in u[1])


def _deps() -> list[str]:
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(
        os.path.join(INCLUDE, "*.h")
    )


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _compile(unit: tuple[str, str, list[str]], extra: list[str]) -> str:
    src, name, flags = unit
    obj = os.path.join(BUILD, name)
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(
        os.path.join(INCLUDE, "*.h")
    )
    if _stale(obj, [src] + headers):
        cmd = [_nvcc(), *ARCH, *NVCC_FLAGS, *flags, *extra, "-I", INCLUDE, "-c", src, "-o", obj + ".tmp"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {name}:\n{r.stderr[-4000:]}")
        os.replace(obj + ".tmp", obj)
    return obj


def build(force: bool = False, extra_flags: list[str] | None = None, jobs: int | None = None) -> str:
    os.makedirs(BUILD, exist_ok=True)
    if not force and not _stale(LIB, _deps()):
        return LIB
    extra = list(extra_flags or [])
    if force:
        for o in glob.glob(os.path.join(BUILD, "*.o")):
            os.remove(o)
    units = _units()
    jobs = jobs or min(len(units), max(1, os.cpu_count() or 1))
    with cf.ThreadPoolExecutor(max_workers=jobs) as ex:
        objs = list(ex.map(lambda u: _compile(u, extra), units))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc(), *ARCH, "-shared", "-cudart", "shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr[-4000:]}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build())
