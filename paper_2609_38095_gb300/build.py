"""Build libzo.so (the C-ABI library) in-tree for sm_103a.

Each .cu file is compiled by its own nvcc process (in parallel), then linked
into one shared library with the CUDA runtime linked statically.
Set ZO_PTXAS_VERBOSE=1 to print register / shared-memory usage.
"""
import concurrent.futures as cf
import os
import platform
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(HERE, "_build", platform.machine())   # objects of this host architecture
LIB = os.path.join(HERE, "libzo.so")
STAMP = LIB + ".arch"   # architecture the library was linked for
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
SOURCES = ["zo_api.cu", "zo_stream_kernels.cu", "zo_update_lut8.cu", "zo_small_kernels.cu",
           "zo_quad_step.cu", "zo_update_items.cu", "zo_update_blocks.cu"]
HEADERS = ["zo_blocks.cuh", "zo_device.cuh", "zo_items.h", "zo_launch.h", "zo_precond.cuh"]


def nvcc() -> str:
    p = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(p):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libzo.so")
    return p


def _flags():
    f = ["-O3", "-std=c++17", "-lineinfo", *ARCH, "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]
    if os.environ.get("ZO_PTXAS_VERBOSE"):
        f += ["-Xptxas", "-v"]
    return f


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(INCLUDE, "zo.h")]
    jobs = []
    objs = []
    for s in SOURCES:
        src = os.path.join(CSRC, s)
        obj = os.path.join(BUILD, s.replace(".cu", ".o"))
        objs.append(obj)
        if force or _stale(obj, [src] + hdrs + [__file__]):
            jobs.append([nvcc(), *_flags(), "-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    if jobs:
        with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
            for cmd, r in ex.map(run, jobs):
                if r.stdout or r.stderr:
                    sys.stderr.write(r.stdout + r.stderr)
                if r.returncode != 0:
                    raise RuntimeError(f"nvcc failed: {' '.join(cmd)}")
    arch_ok = os.path.exists(STAMP) and open(STAMP).read().strip() == platform.machine()
    if force or jobs or not arch_ok or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc(), *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed: {r.stderr}")
        os.replace(tmp, LIB)
        with open(STAMP, "w") as f:
            f.write(platform.machine())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv))
