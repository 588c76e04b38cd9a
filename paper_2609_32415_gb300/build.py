"""Build librefadapt.so (the C-ABI library) in-tree with nvcc for sm_103a, and
_binding.so, the Python binding's native argument marshalling.

Each .cu under csrc/ is compiled in parallel to an object file, then all are
linked into paper_2609_32415_gb300/librefadapt.so (static CUDA runtime, no
torch dependency). csrc/binding.cpp is compiled with the host compiler against
the installed torch's headers meanwhile and linked to that library. Rebuilds
only when a source or header is newer than the libraries, or when _binding.so was
made for another torch or Python than the ones that run.
"""
import glob
import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "librefadapt.so")
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
BINDING = os.path.join(PKG, "_binding.so")
BINDING_FOR = os.path.join(BUILD_DIR, "binding.for")  # what _binding.so was made for
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the RefAdapt CUDA library cannot be built")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + [BINDING_SRC] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]


def _binding_for() -> str:
    import torch
    return "torch %s, %s" % (torch.__version__, sys.implementation.cache_tag)


def up_to_date() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(BINDING) or not os.path.exists(BINDING_FOR):
        return False
    with open(BINDING_FOR) as f:
        if f.read() != _binding_for():
            return False
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    return all(os.path.getmtime(f) <= t for f in _deps())


def _compile_binding() -> str:
    """csrc/binding.cpp -> object file (host compiler, the installed torch's headers)."""
    import sysconfig

    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    obj = os.path.join(BUILD_DIR, "binding.o")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-I", INCLUDE]
    for d in (inc, os.path.join(inc, "torch", "csrc", "api", "include"), cuda, sysconfig.get_paths()["include"]):
        cmd += ["-isystem", d]
    _run(cmd + ["-c", BINDING_SRC, "-o", obj], "compiling binding.cpp")
    return obj


def _run(cmd, what):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("%s failed" % what)


def _link_binding(obj):
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = BINDING + ".tmp.%d" % os.getpid()
    _run([os.environ.get("CXX", "g++"), "-shared", "-o", tmp, obj, "-L", PKG, "-l:librefadapt.so", "-Wl,-rpath,$ORIGIN",
          "-L", lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"], "linking _binding.so")
    os.replace(tmp, BINDING)
    with open(BINDING_FOR, "w") as f:
        f.write(_binding_for())


def build(force: bool = False, verbose: bool = False, extra_flags=None) -> str:
    """Compile csrc/*.cu and link librefadapt.so; return the library path."""
    if not force and up_to_date():
        return LIB
    nvcc = _nvcc()
    os.makedirs(BUILD_DIR, exist_ok=True)
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
                    "--expt-relaxed-constexpr"] + list(extra_flags or [])
    srcs = _sources()

    def compile_one(src):
        obj = os.path.join(BUILD_DIR, os.path.basename(src) + ".o")
        cmd = [nvcc] + flags + ["-c", src, "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed on %s" % os.path.basename(src))
        return obj

    with ThreadPoolExecutor(max_workers=max(1, min(len(srcs) + 1, os.cpu_count() or 1))) as ex:
        binding = ex.submit(_compile_binding)
        objs = list(ex.map(compile_one, srcs))
        binding_obj = binding.result()
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("linking librefadapt.so failed")
    os.replace(tmp, LIB)
    _link_binding(binding_obj)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
