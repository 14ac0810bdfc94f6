"""Builds libcover.so (the C-ABI kernel library) in-tree with nvcc for sm_103a, and beside it
_binding.so (the Python calls' native argument marshalling) with the host compiler.

Each translation unit compiles in parallel; the objects link into
``paper_2602_06161_gb300/libcover.so``. The CUDA runtime is linked statically
and the driver is reached only through cudaGetDriverEntryPointByVersion, so
the library loads on machines without a GPU driver.

libcover.so depends on neither PyTorch nor the interpreter; _binding.so is compiled against the
headers of both, and is made again when either is another one. Where it cannot be made (no Python
headers, say), the calls are marshalled in Python.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import warnings

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libcover.so")
BINDING = os.path.join(PKG, "_binding.so")
BINDING_TAG = os.path.join(BUILD, "binding.tag")   # what _binding.so was compiled for, or failed to be

SOURCES = ["cover_api.cu", "context.cu", "tmap.cu", "route_kernel.cu", "attn_f32.cu", "attn_bf16_sm103.cu", "attn_window_gqa.cu",
           "score_kernel.cu", "kv_kernel.cu", "mass_kernel.cu", "debug_kernels.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _newer(deps, than: str) -> bool:
    t = os.path.getmtime(than)
    return any(os.path.getmtime(d) > t for d in deps)


def _stale() -> bool:
    """Whether libcover.so is missing or older than its sources."""
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "binding.cpp"] + [
        os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)] + [os.path.abspath(__file__)]
    return not os.path.exists(LIB) or _newer(deps, LIB)


def _binding_tag() -> str:
    """The PyTorch build and the interpreter whose headers _binding.so is compiled against."""
    import sysconfig

    import torch

    return " ".join([torch.__version__, str(torch.version.git_version), str(int(torch._C._GLIBCXX_USE_CXX11_ABI)),
                     sysconfig.get_config_var("EXT_SUFFIX"), sys.version.split()[0]])


def _binding_stale() -> bool:
    """Whether _binding.so has to be made: it is missing (and not known to fail), older than its sources, or
    was compiled for another PyTorch or interpreter, whose objects it would read by a layout that they lack."""
    try:
        with open(BINDING_TAG) as f:
            made_for = f.read()
    except OSError:
        return True
    if made_for != _binding_tag() + ("" if os.path.exists(BINDING) else " failed"):
        return True
    return _newer([os.path.join(CSRC, "binding.cpp"), os.path.join(INCLUDE, "cover.h"), os.path.abspath(__file__)],
                  BINDING_TAG)


def _compile_binding(tmp: str) -> None:
    import sysconfig

    import torch

    root = os.path.dirname(torch.__file__)
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for inc in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                os.path.join(os.path.dirname(os.path.dirname(nvcc())), "include"), sysconfig.get_paths()["include"]):
        cmd += ["-isystem", inc]
    lib = os.path.join(root, "lib")
    cmd += ["-I", INCLUDE, os.path.join(CSRC, "binding.cpp"), "-o", tmp, "-L" + lib, "-Wl,-rpath," + lib,
            "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
    except OSError as e:
        raise RuntimeError(f"binding.cpp failed: {e}") from e
    if r.returncode != 0:
        raise RuntimeError(f"binding.cpp failed:\n{r.stdout}\n{r.stderr}")


def _build_binding() -> None:
    """Makes _binding.so. A failure leaves none (never one of another PyTorch) and a warning."""
    tag, tmp = _binding_tag(), BINDING + ".tmp"
    try:
        os.makedirs(BUILD, exist_ok=True)
        try:
            _compile_binding(tmp)
            os.replace(tmp, BINDING)
        except RuntimeError as e:
            if os.path.exists(BINDING):
                os.remove(BINDING)
            tag += " failed"
            warnings.warn(f"the native argument marshalling could not be built, calls are marshalled in Python: {e}")
        with open(BINDING_TAG, "w") as f:
            f.write(tag)
    except OSError as e:   # a tree that cannot be written to: without the tag the object is not used
        warnings.warn(f"the native argument marshalling could not be built, calls are marshalled in Python: {e}")


def build(force: bool = False, verbose_ptxas: bool = False, quiet: bool = True) -> str:
    """Compile what is stale and return the path of libcover.so."""
    lib, binding = force or _stale(), force or _binding_stale()
    with cf.ThreadPoolExecutor(max_workers=1) as ex:
        made = ex.submit(_build_binding) if binding else None
        if lib:
            _build_lib(verbose_ptxas, quiet)
        if made is not None:
            made.result()
    return LIB


def _build_lib(verbose_ptxas: bool, quiet: bool) -> None:
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()

    def compile_one(src: str):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        cmd = [cc, *ARCH, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose_ptxas:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        return src, obj, r

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    logs = []
    for src, obj, r in results:
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if r.stderr.strip():
            logs.append(f"--- {src}\n{r.stderr}")
    tmp = LIB + ".tmp"
    cmd = [cc, *ARCH, "-shared", "-o", tmp, *[o for _, o, _ in results], "-cudart", "static"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    if logs and (verbose_ptxas or not quiet):
        print("\n".join(logs), file=sys.stderr)


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose_ptxas="-v" in sys.argv, quiet=False)
    print(LIB)
