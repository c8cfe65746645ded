"""Builds libsparkattn.so in-tree with nvcc for sm_100a (no JIT cache, no torch headers), and _sparkattn.so, the binding's
native argument marshalling, with the host compiler against torch's headers."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsparkattn.so")
BINDING = os.path.join(HERE, "_sparkattn.so")
OBJDIR = os.path.join(HERE, "build")
BINDING_FOR = os.path.join(OBJDIR, "_sparkattn.for")      # what the binding was built against
SOURCES = ["api.cu", "select.cu", "quant.cu", "fwd.cu", "noalloc.cu", "comp.cu", "fwd_pipe.cu", "reorder.cu"]
NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _target() -> str:
    """The torch and Python that a binding built now belongs to: it uses torch's C++ interface, which is another one in
    every build of torch, and Python's."""
    import torch
    return f"torch {torch.__version__} {torch.version.git_version} python {sysconfig.get_config_var('SOABI')}"


def _binding_target() -> str:
    try:
        with open(BINDING_FOR) as f:
            return f.read()
    except FileNotFoundError:
        return ""


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(BINDING) or _binding_target() != _target():
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "sparkattn.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = _nvcc()
    os.makedirs(OBJDIR, exist_ok=True)

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJDIR, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        return obj

    def build_binding() -> None:
        import torch
        root = os.path.dirname(torch.__file__)
        cuda = os.path.dirname(os.path.dirname(nvcc)) if os.path.sep in nvcc else "/usr/local/cuda"
        inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
               *("-I" + i for i in inc), os.path.join(CSRC, "binding.cpp"), "-o", BINDING,
               "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("g++ failed on binding.cpp")
        with open(BINDING_FOR, "w") as f:
            f.write(_target())

    with ThreadPoolExecutor(max_workers=5) as ex:
        binding = ex.submit(build_binding)
        objs = list(ex.map(compile_one, SOURCES))
        binding.result()
    cmd = [nvcc, "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
