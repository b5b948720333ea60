"""In-tree build of libdust.so for sm_103a (nvcc, no cmake) and of _front, the
front end's native half (g++, against the installed torch's headers).

Each .cu under csrc/ is compiled to an object in parallel, then linked into
paper_0907_3768_gb300/_build/libdust.so with the CUDA runtime linked
statically (the library then needs only the driver at run time).
"""
import concurrent.futures as cf
import contextlib
import glob
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libdust.so")
FRONT_SRC = os.path.join(CSRC, "front.cpp")
FRONT = os.path.join(OUT, "_front" + sysconfig.get_config_var("EXT_SUFFIX"))
FRONT_STAMP = FRONT + ".built_against"
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr", "-I" + INCLUDE]


def nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))


def up_to_date():
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in _deps())


def front_built_against():
    """What a _front module holds for: the torch whose headers, ABI and libraries it was compiled against."""
    import torch

    return f"torch {torch.__version__} in {os.path.dirname(torch.__file__)}, C++11 ABI {int(torch._C._GLIBCXX_USE_CXX11_ABI)}\n"


def front_up_to_date():
    if not (os.path.exists(FRONT) and os.path.exists(FRONT_STAMP)):
        return False
    t = os.path.getmtime(FRONT)
    if any(os.path.getmtime(p) > t for p in (FRONT_SRC, os.path.join(INCLUDE, "dust.h"), os.path.abspath(__file__))):
        return False
    with open(FRONT_STAMP) as f:
        return f.read() == front_built_against()


def build_front(force=False):
    """Compile and link the _front module; returns its path."""
    if not force and front_up_to_date():
        return FRONT
    import torch
    from torch.utils import cpp_extension

    os.makedirs(OUT, exist_ok=True)
    for old in (FRONT_STAMP, FRONT):  # a module of another torch must not stay where this build fails
        with contextlib.suppress(FileNotFoundError):
            os.remove(old)
    inc = [*cpp_extension.include_paths("cuda"), "/usr/local/cuda/include", sysconfig.get_path("include")]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = FRONT + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *["-I" + p for p in inc], FRONT_SRC, "-o", tmp, "-L" + lib, "-Wl,-rpath," + lib,
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on front.cpp:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, FRONT)
    with open(FRONT_STAMP + f".tmp{os.getpid()}", "w") as f:
        f.write(front_built_against())
    os.replace(f.name, FRONT_STAMP)
    return FRONT


def build(force=False, verbose=False, ptxas_verbose=False):
    """Compile and link libdust.so and the _front module; returns libdust.so's path.
    Where _front cannot be built (no torch headers, another ABI) that is a warning: the Python
    front end works without it."""
    with cf.ThreadPoolExecutor(max_workers=1) as ex:
        front = ex.submit(build_front, force)
        lib = build_lib(force, verbose, ptxas_verbose)
        try:
            front.result()
        except (RuntimeError, ImportError, OSError) as e:
            warnings.warn(f"the front end's native half was not built: {e}", RuntimeWarning, stacklevel=2)
    return lib


def build_lib(force=False, verbose=False, ptxas_verbose=False):
    """Compile and link libdust.so; returns its path."""
    if not force and up_to_date():
        return LIB
    os.makedirs(os.path.join(OUT, "obj"), exist_ok=True)
    cc = nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_verbose else []

    def compile_one(src):
        obj = os.path.join(OUT, "obj", os.path.basename(src) + ".o")
        cmd = [cc, *ARCH, *FLAGS, *extra, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stdout + r.stderr

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as ex:
        results = list(ex.map(compile_one, sources()))
    if verbose or ptxas_verbose:
        for _, log in results:
            if log.strip():
                print(log, file=sys.stderr)
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [cc, *ARCH, "-shared", "-o", tmp, *[o for o, _ in results], "-cudart", "static"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_verbose="--ptxas" in sys.argv))
