"""Build the C-ABI CUDA library for sm_100a with nvcc and the Python binding's native side with the
host compiler, in-tree, next to this file."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgdn_b200.so")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "--threads", "0"]
BINDING_SRC = os.path.join(HERE, "binding", "binding.cpp")
BINDING = os.path.join(HERE, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))
CXX_FLAGS = ["-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newer(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _headers():
    return glob.glob(os.path.join(HERE, "..", "include", "*.h"))


def is_stale() -> bool:
    return _newer(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())


def binding_key() -> str:
    """What the binding is compiled against besides its sources.  It goes into the module as a string, so that one
    built for another torch is found stale however old or new its file is."""
    import torch
    return f"gdn-binding-key:torch-{torch.__version__}-{torch.version.git_version}:abi-{int(torch._C._GLIBCXX_USE_CXX11_ABI)};"


def binding_is_stale() -> bool:
    if _newer(BINDING, [BINDING_SRC, *_headers()]):
        return True
    with open(BINDING, "rb") as f:
        return binding_key().encode() not in f.read()


def _build_binding() -> None:
    """The extension module links against the library next to it and against the torch libraries
    that `import torch` has loaded."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = BINDING + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++")] + CXX_FLAGS + [f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                                                              f'-DGDN_BINDING_KEY="{binding_key()}"']
    for inc in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                sysconfig.get_paths()["include"], os.path.join(cuda, "include")):
        cmd += ["-isystem", inc]
    cmd += [BINDING_SRC, "-o", tmp, "-L" + HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN",
            "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.check_call(cmd)
    os.replace(tmp, BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or is_stale():
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + sources() + ["-o", tmp]
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    if force or binding_is_stale():
        _build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
