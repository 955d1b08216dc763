"""Device functions of the library's headers, called on their own: a small CUDA
source that includes them is compiled with the library's flags and loaded."""
import ctypes
import os
import subprocess

import torch

from paper_1705_03666_gb300 import build


def load(tmp_path, source: str) -> ctypes.CDLL:
    src, lib = os.path.join(tmp_path, "part.cu"), os.path.join(tmp_path, "part.so")
    with open(src, "w") as f:
        f.write(source)
    cmd = [build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-Xcompiler", "-fvisibility=default",
           "-I", build.CSRC, "-shared", "-o", lib, src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(lib)


def call(fn, *args):
    """fn(*args) with tensors as their device pointers; waits, and checks the
    cudaError_t that it returns."""
    conv = [ctypes.c_void_p(a.data_ptr()) if isinstance(a, torch.Tensor) else a for a in args]
    torch.cuda.synchronize()
    assert fn(*conv) == 0
    torch.cuda.synchronize()
