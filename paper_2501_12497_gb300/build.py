"""Build libmof.so for sm_103a from csrc/*.cu with nvcc and the autograd nodes of
csrc/autograd.cpp with the C++ compiler (parallel compile, in tree).

Output: paper_2501_12497_gb300/_build/libmof.so and _autograd.so beside it. Re-run is a
no-op unless a source or header is newer than what was built from it, or _autograd.so was built
for another torch or Python. libmof.so needs neither and is linked whatever becomes of the nodes.
"""
import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(HERE, "_build")
LIB_PATH = os.path.join(BUILD_DIR, "libmof.so")
AUTOGRAD_SRC = os.path.join(CSRC, "autograd.cpp")
AUTOGRAD_PATH = os.path.join(BUILD_DIR, "_autograd.so")
AUTOGRAD_FOR = os.path.join(BUILD_DIR, "_autograd.for")  # what _autograd.so was built for
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
         "-I" + INCLUDE, "-I" + CSRC]


def _nvcc():
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found; the CUDA toolkit is required to build libmof")
    return cand


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps():
    files = sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    files.append(os.path.join(INCLUDE, "mof.h"))
    return files


def _run(cmd, what, verbose=False):
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0 or verbose:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError("%s failed" % what)


def _stale(out, deps, force):
    return force or not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(f) for f in deps)


def _torch_id():
    """The torch and Python in use, without importing torch."""
    spec = importlib.util.find_spec("torch")
    version = os.path.join(os.path.dirname(spec.origin), "version.py") if spec and spec.origin else ""
    text = open(version).read() if os.path.exists(version) else ""
    return "%s\n%s\n%s" % (sysconfig.get_config_var("SOABI"), version, text)


def _read(path):
    return open(path).read() if os.path.exists(path) else None


def _compile_autograd(obj, verbose):
    import torch  # here, as the CUDA library alone needs none of it
    t = os.path.join(os.path.dirname(torch.__file__), "include")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    incs = [INCLUDE, t, os.path.join(t, "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
            os.path.join(cuda, "include")]
    cmd = ["g++", "-c", AUTOGRAD_SRC, "-o", obj, "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi())] + ["-I" + i for i in incs]
    _run(cmd, "compilation of autograd.cpp", verbose)
    return os.path.join(os.path.dirname(torch.__file__), "lib")


def build(force=False, verbose=False, extra=()):
    """Compile every translation unit and link libmof.so and _autograd.so; returns libmof.so's path."""
    os.makedirs(BUILD_DIR, exist_ok=True)
    lib = _stale(LIB_PATH, _deps(), force)
    bind_for = _torch_id()
    bind = _stale(AUTOGRAD_PATH, [AUTOGRAD_SRC, os.path.join(INCLUDE, "mof.h")], force) or _read(AUTOGRAD_FOR) != bind_for
    if not lib and not bind:
        return LIB_PATH
    nvcc = _nvcc()
    pid = os.getpid()
    objs = [os.path.join(BUILD_DIR, os.path.basename(f)[:-3] + ".o") for f in sources()]
    obj = os.path.join(BUILD_DIR, "autograd.o")
    with ThreadPoolExecutor(max_workers=max(2, min(9, os.cpu_count() or 4))) as ex:
        nodes = ex.submit(_compile_autograd, obj, verbose) if bind else None
        jobs = [ex.submit(_run, [nvcc, "-c", f, "-o", o] + ARCH + FLAGS + list(extra), "nvcc on %s" % f, verbose)
                for f, o in zip(sources(), objs)] if lib else []
        for j in jobs:
            j.result()
        if lib:
            tmp = LIB_PATH + ".tmp%d" % pid
            _run([nvcc, "-shared", "-o", tmp] + objs + ARCH, "link of libmof.so")
            os.replace(tmp, LIB_PATH)
        if bind:
            torch_lib = nodes.result()
            tmp = AUTOGRAD_PATH + ".tmp%d" % pid
            _run(["g++", "-shared", "-o", tmp, obj, "-L" + torch_lib, "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu",
                  "-ltorch_cuda", "-ltorch_python", "-L" + BUILD_DIR, "-l:libmof.so", "-Wl,-rpath,$ORIGIN"], "link of _autograd.so")
            os.replace(tmp, AUTOGRAD_PATH)
            with open(tmp, "w") as f:
                f.write(bind_for)
            os.replace(tmp, AUTOGRAD_FOR)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
