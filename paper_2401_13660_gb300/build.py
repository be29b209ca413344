"""Build libmbscan.so (the C-ABI CUDA library) in-tree for sm_103a, and the
native part of its Python binding.

Each .cu under csrc/ is compiled to an object file by nvcc (in parallel),
then linked into _build/libmbscan.so with the CUDA runtime linked statically,
so the library loads on a machine without a GPU (for the export checks) and
needs nothing but the driver on a GPU machine. csrc/binding.cpp (argument
marshalling on torch tensors) is compiled by g++ into a module beside it, named
after the Python and torch it was built for; only that file depends on torch.
Where it cannot be built the library is complete without it: mbscan.py then
marshals in Python.

    python -m paper_2401_13660_gb300.build [--force] [--verbose]
"""
from __future__ import annotations

import argparse
import concurrent.futures as cf
import hashlib
import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.environ.get("MBSCAN_BUILD_DIR") or os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libmbscan.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")


def torch_dir():
    """Directory of the installed torch, found without importing it (None: not installed)."""
    spec = importlib.util.find_spec("torch")
    return os.path.dirname(spec.origin) if spec and spec.origin else None


def binding_path() -> str:
    """The binding for this Python and torch: a module built for others has another name and is never loaded."""
    version = b""
    if torch_dir():
        with open(os.path.join(torch_dir(), "version.py"), "rb") as f:   # torch's version and the commit it was built from
            version = f.read()
    return os.path.join(BUILD, f"_mbcall.{sysconfig.get_config_var('SOABI')}."
                               f"torch-{hashlib.sha256(version).hexdigest()[:12]}.so")


BINDING = binding_path()

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC,-O2",
              "--expt-relaxed-constexpr", "-I", INCLUDE]
# Extra nvcc flags (e.g. -D tuning macros) for builds into MBSCAN_BUILD_DIR.
NVCC_FLAGS += os.environ.get("MBSCAN_NVCC_FLAGS", "").split()


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found (set NVCC or put CUDA's bin/ on PATH)")


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps():
    return sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC)
                        if f.endswith((".cuh", ".h", ".cpp"))] + [os.path.join(INCLUDE, "mbscan.h")]


def _newer(path) -> bool:
    """Whether `path` exists and is newer than every source."""
    return os.path.exists(path) and all(os.path.getmtime(d) <= os.path.getmtime(path) for d in _deps())


def up_to_date() -> bool:
    """Whether the library is, and the binding or the note that it could not be built."""
    return _newer(LIB) and (_newer(BINDING) or _newer(BINDING + ".failed"))


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
    cmd = [nvcc(), *ARCH, *NVCC_FLAGS, "-c", src, "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
    if verbose and r.stderr:
        sys.stderr.write(r.stderr)
    return obj


def _compile_binding() -> str:
    """Compile the binding; what went wrong, or an empty string."""
    try:
        if not torch_dir():
            return "torch is not installed"
        cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc())))
        inc = [INCLUDE, sysconfig.get_paths()["include"], os.path.join(torch_dir(), "include"),
               os.path.join(torch_dir(), "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
        tmp = BINDING + f".tmp{os.getpid()}"
        cmd = ["g++", "-O2", "-std=c++20", "-fPIC", "-shared", *(f"-I{d}" for d in inc),
               os.path.join(CSRC, "binding.cpp"), "-o", tmp, f"-L{os.path.join(torch_dir(), 'lib')}",
               "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            return f"g++ failed on binding.cpp:\n{r.stdout}\n{r.stderr}"
        os.replace(tmp, BINDING)
        return ""
    except OSError as e:   # no g++, ...
        return str(e)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel for sm_103a and link libmbscan.so; returns its path."""
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    srcs = sources()
    with cf.ThreadPoolExecutor(max_workers=min(12, len(srcs) + 1)) as ex:
        binding = ex.submit(_compile_binding)
        objs = list(ex.map(lambda s: _compile(s, verbose), srcs))
        wrong = binding.result()
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    note = BINDING + ".failed"   # not tried again until a source changes
    if wrong:
        with open(note, "w") as f:
            f.write(wrong)
        warnings.warn(f"native argument marshalling not built, calls are marshalled in Python: {wrong}")
    elif os.path.exists(note):
        os.remove(note)
    return LIB


if __name__ == "__main__":
    ap = argparse.ArgumentParser()
    ap.add_argument("--force", action="store_true")
    ap.add_argument("--verbose", action="store_true", help="print ptxas register/smem usage")
    a = ap.parse_args()
    print(build(force=a.force, verbose=a.verbose))
