"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libscap_b200.so")
# the binding's call helper, named for the interpreter it is built against: another one does not load it
CALL = os.path.join(HERE, "_scap_call" + sysconfig.get_config_var("EXT_SUFFIX"))

# no --use_fast_math: the mask arithmetic must round exactly as documented
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def _newer(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu to an object (in parallel) and link libscap_b200.so; a no-op when up to date."""
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdrs = _headers()
    jobs = []
    objs = []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _newer(obj, [src] + hdrs):
            cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
            if verbose:
                cmd[1:1] = ["-Xptxas", "-v"]
            jobs.append(cmd)
    if jobs:
        with cf.ThreadPoolExecutor(len(jobs)) as ex:
            for cmd, rc in zip(jobs, ex.map(lambda c: subprocess.run(c).returncode, jobs)):
                if rc != 0:
                    raise RuntimeError("nvcc failed: " + " ".join(cmd))
    if jobs or force or _newer(LIB, objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "--shared", "-cudart", "static",
                               "-o", tmp, *objs])
        os.replace(tmp, LIB)
    build_call_helper(force)
    return LIB


def build_call_helper(force: bool = False, target: str = CALL) -> bool:
    """The binding's call helper.  It needs a C compiler and the Python headers; without them the CUDA library is complete all the
    same and the binding calls it through ctypes, so a failure here is reported and no more."""
    src = os.path.join(CSRC, "scap_pycall.c")
    if not force and not _newer(target, [src]):
        return True
    tmp = target + ".tmp.%d" % os.getpid()
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], src, "-o", tmp]
    try:
        subprocess.check_call(cmd)
    except (OSError, subprocess.CalledProcessError) as e:
        print("the call helper was not built (%s): calls go through ctypes, about 5 us slower each" % e, file=sys.stderr)
        return False
    os.replace(tmp, target)
    return True


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
