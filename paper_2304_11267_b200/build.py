"""Build the C-ABI attention library (nvcc, sm_100a) and its torch binding (g++) in-tree; neither needs a GPU."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libsd_attn.so")
EXT = os.path.join(PKG, "_sd_torch.so")
EXT_SOURCE = os.path.join(CSRC, "torch_binding.cpp")
INCLUDE = os.path.join(os.path.dirname(PKG), "include")

NVCC_FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
              "--compiler-options", "-fPIC", "-shared", "-cudart", "shared"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [EXT_SOURCE] if target == EXT else [f for f in glob.glob(os.path.join(CSRC, "*")) if f != EXT_SOURCE]
    return any(os.path.getmtime(f) > t for f in deps + glob.glob(os.path.join(INCLUDE, "*.h")))


def _compile(cmd, target: str, verbose: bool) -> None:
    """Run the compiler into a temporary file and put it in the target's place."""
    tmp = target + ".tmp.%d" % os.getpid()
    proc = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
    if proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
        raise RuntimeError("%s failed building %s" % (os.path.basename(cmd[0]), os.path.basename(target)))
    if verbose:
        sys.stderr.write(proc.stdout + proc.stderr)
    os.replace(tmp, target)


def _extension_command():
    import torch
    base = os.path.dirname(torch.__file__)
    include = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
               os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"), sysconfig.get_paths()["include"]]
    lib = os.path.join(base, "lib")
    return (["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden",
             "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi())] +
            [a for d in include for a in ("-isystem", d)] + [EXT_SOURCE, "-L", PKG, "-l:libsd_attn.so", "-L", lib] +
            ["-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"])


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libsd_attn.so and csrc/torch_binding.cpp into _sd_torch.so next to this file; returns the
    library's path."""
    if force or _stale(LIB):
        _compile([_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-I", INCLUDE] + sources(), LIB, verbose)
    if force or _stale(EXT):
        _compile(_extension_command(), EXT, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
