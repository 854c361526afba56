"""In-tree build of the C-ABI CUDA library (libsmartgen.so) for sm_100a with nvcc.

Each csrc/*.cu is compiled to an object under build/ (in parallel, skipped when up to date) and
the objects are linked into paper_2607_28150_b200/libsmartgen.so with the CUDA runtime linked
statically, so the library loads on a machine without a GPU or a driver.  csrc/native.cpp, the marshalling
between torch tensors and the library, becomes the extension module _native (with the interpreter's suffix) beside it.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJDIR = os.path.join(ROOT, "build", "obj")
LIB = os.path.join(HERE, "libsmartgen.so")
EXT_SUFFIX = sysconfig.get_config_var("EXT_SUFFIX")          # names the interpreter
NATIVE = os.path.join(HERE, "_native" + EXT_SUFFIX)

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--use_fast_math", "-I", INCLUDE, "-I", CSRC,
]


# Extra nvcc flags for a debug or profiling build of the whole library, e.g. SG_NVCC_FLAGS="-DSG_SCORE_PROFILE";
# such a build always recompiles, and so does the next ordinary one.
EXTRA_FLAGS = os.environ.get("SG_NVCC_FLAGS", "").split()
_STAMP = os.path.join(OBJDIR, "flags.txt")


def _nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return cand


def _newest_dep() -> float:
    deps = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]
    return max(os.path.getmtime(p) for p in deps)


def _compile(src: str, obj: str, verbose: bool) -> None:
    cmd = [_nvcc()] + NVCC_FLAGS + EXTRA_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, res.stdout, res.stderr))
    if verbose:
        sys.stderr.write(res.stderr)


def native_stamp() -> str:
    """What the extension module is compiled against: it reads tensors through inline code of torch's headers, so it fits
    one version of torch and one interpreter.  The module carries the stamp (BUILT_FOR)."""
    import torch
    return "built for torch %s, CUDA %s, C++11 ABI %d, Python %s" % (torch.__version__, torch.version.cuda,
                                                                    int(torch.compiled_with_cxx11_abi()), EXT_SUFFIX)


def native_is_current() -> bool:
    src = os.path.join(CSRC, "native.cpp")
    newest = max(os.path.getmtime(p) for p in (src, os.path.join(CSRC, "internal.h"), os.path.join(INCLUDE, "smartgen.h"), os.path.abspath(__file__)))
    if not os.path.exists(NATIVE) or os.path.getmtime(NATIVE) < newest:
        return False
    with open(NATIVE, "rb") as f:
        return native_stamp().encode() in f.read()


def _build_native(force: bool) -> None:
    plain = os.path.join(HERE, "_native.so")                 # a module without the interpreter's suffix would be imported by any
    if os.path.exists(plain):
        os.remove(plain)
    if not force and native_is_current():
        return
    src = os.path.join(CSRC, "native.cpp")
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi()),
           "-DSG_BUILT_FOR=\"%s\"" % native_stamp(), "-I", INCLUDE,
           "-isystem", inc, "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
           "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"), src, "-o", tmp,
           "-L", HERE, "-l:libsmartgen.so", "-L", lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
           "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("building the marshalling module failed:\n%s\n%s" % (res.stdout, res.stderr))
    os.replace(tmp, NATIVE)


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    if not srcs:
        raise RuntimeError("no CUDA sources under %s" % CSRC)
    os.makedirs(OBJDIR, exist_ok=True)
    last = open(_STAMP).read() if os.path.exists(_STAMP) else ""
    if last != " ".join(EXTRA_FLAGS):
        force = True                                     # objects on disk were built with other flags
    dep_time = _newest_dep()
    jobs, objs = [], []
    for s in srcs:
        o = os.path.join(OBJDIR, os.path.basename(s)[:-3] + ".o")
        objs.append(o)
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(os.path.getmtime(s), dep_time):
            jobs.append((s, o))
    if jobs:
        with concurrent.futures.ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            list(ex.map(lambda so: _compile(so[0], so[1], verbose), jobs))
    if jobs or not os.path.exists(LIB) or any(os.path.getmtime(o) > os.path.getmtime(LIB) for o in objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        cmd = [_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static",
               "-o", tmp] + objs
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("link failed:\n%s\n%s" % (res.stdout, res.stderr))
        os.replace(tmp, LIB)
    _build_native(force)
    with open(_STAMP, "w") as f:
        f.write(" ".join(EXTRA_FLAGS))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
