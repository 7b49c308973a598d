"""Build the C-ABI shared library `libexmoe.so` (nvcc, sm_100a) and its CPython module `_exmoe_native.so` (g++) in-tree.

    python -m paper_2608_15383_b200.build [--force] [--verbose]
"""
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libexmoe.so")
NATIVE = os.path.join(PKG, "_exmoe_native.so")
NATIVE_SOURCE = "binding_native.cpp"
SOURCES = ["pack.cu", "plan.cu", "decode.cu", "stream.cu", "prefill.cu", "tcstream.cu", "route.cu", "cache.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--shared", "--threads", "8"]


def _stale(target, sources):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in sources] + [os.path.join(PKG, "..", "include", "exmoe.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _torch_tag():
    import torch
    return f"built for torch {torch.__version__}"


def native_is_current(path=NATIVE):
    """Whether the CPython module at `path` was built for the torch of this process (it says so in a string of its own)."""
    with open(path, "rb") as f:
        return _torch_tag().encode() + b"\0" in f.read()


def _run(cmd, verbose, target):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode:
        raise RuntimeError(f"building {os.path.basename(target)} failed")


def build(force=False, verbose=False):
    """Compile csrc/ into libexmoe.so and _exmoe_native.so (cross-compiles without a GPU).  Returns the library's path."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if force or _stale(LIB, [f for f in os.listdir(CSRC) if f != NATIVE_SOURCE]):
        extra = os.environ.get("EXMOE_NVCC_EXTRA", "").split()      # e.g. -DEXMOE_DISABLE_PDL for an A/B timing
        _run([nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) +
             [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB, "-lcudart"], verbose, LIB)
    if force or _stale(NATIVE, [NATIVE_SOURCE]) or not native_is_current():
        import torch
        from torch.utils.cpp_extension import include_paths
        libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
        inc = [f"-I{d}" for d in include_paths() + [sysconfig.get_paths()["include"], cuda]]
        _run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f'-DEXMOE_TORCH_TAG="{_torch_tag()}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] +
             inc + [os.path.join(CSRC, NATIVE_SOURCE), "-o", NATIVE, f"-L{libdir}", "-ltorch_python", "-ltorch_cuda",
                    "-ltorch_cpu", "-lc10_cuda", "-lc10"], verbose, NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
