"""The native marshalling reads the tensors' sizes before it lets other Python threads run.  binding.cpp is
built against stand-ins for the library's entry points that record the sizes they are given, with CPU tensors passing
for CUDA ones and a callback at the point where the interpreter lock is released, which does what another thread
might: it reshapes the tensors of the call."""
import ctypes
import importlib.util
import os
import subprocess
import sysconfig

import pytest
import torch

PACKAGE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200")

STAND_IN = r"""
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#undef Py_BEGIN_ALLOW_THREADS
#undef Py_END_ALLOW_THREADS
extern "C" void lock_released();
#define Py_BEGIN_ALLOW_THREADS { lock_released();
#define Py_END_ALLOW_THREADS }
#define is_cuda is_cpu
namespace c10::cuda {
struct NoStream { void* stream() const { return nullptr; } };
inline NoStream no_stream() { return {}; }
}
#define getCurrentCUDAStream no_stream
"""

RECORDER = r"""
#include "%(root)s/include/gdn.h"
#define EXPORT __attribute__((visibility("default")))
extern "C" {
EXPORT int seen[8];
EXPORT PyObject* callback = nullptr;
void lock_released() {
    PyObject* r = PyObject_CallNoArgs(callback);
    Py_XDECREF(r);
}
static int record(std::initializer_list<int> sizes) {
    int i = 0;
    for (int s : sizes) seen[i++] = s;
    return 0;
}
int gdn_decode(const void*, const void*, const void*, const float*, const float*, float*, const int32_t*, void*, int32_t B,
               int32_t Hqk, int32_t Hv, int32_t dk, int32_t dv, int32_t slots, float, int32_t*, void*) {
    return record({B, Hqk, Hv, dk, dv, slots});
}
int gdn_decode_multi(const void*, const void*, const void*, const float*, const float*, float*, const int32_t*, void*,
                     int32_t B, int32_t L, int32_t Hqk, int32_t Hv, int32_t dk, int32_t dv, int32_t slots, float, int32_t,
                     int32_t*, void*) {
    return record({B, L, Hqk, Hv, dk, dv, slots});
}
int gdn_gate(const void*, const void*, const float*, const float*, float*, float*, int32_t T, int32_t Hv, void*) {
    return record({T, Hv});
}
#define PREFILL(name) \
    int name(const void*, const void*, const void*, const float*, const float*, const int32_t*, const float*, float*, \
             const int32_t*, void*, int32_t T, int32_t N, int32_t, int32_t Hqk, int32_t Hv, int32_t dk, int32_t dv, int32_t, \
             int32_t slots, float, void*, size_t, int32_t*, void* EXTRA) { \
        return record({T, N, Hqk, Hv, dk, dv, slots}); \
    }
#define EXTRA
PREFILL(gdn_prefill) PREFILL(gdn_prefill_chunked) PREFILL(gdn_prefill_fused) PREFILL(gdn_prefill_stream)
#undef EXTRA
#define EXTRA , int32_t
PREFILL(gdn_prefill_overlap)
}
"""


@pytest.fixture(scope="module")
def recorder(tmp_path_factory):
    d = tmp_path_factory.mktemp("binding")
    (d / "stand_in.h").write_text(STAND_IN)
    (d / "recorder.cpp").write_text(RECORDER % {"root": os.path.dirname(PACKAGE)})
    root = os.path.dirname(torch.__file__)
    out = str(d / ("_binding" + sysconfig.get_config_var("EXT_SUFFIX")))
    cmd = ["g++", "-O0", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-include", str(d / "stand_in.h")]
    for inc in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                sysconfig.get_paths()["include"], os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")):
        cmd += ["-isystem", inc]
    cmd += [os.path.join(PACKAGE, "binding", "binding.cpp"), str(d / "recorder.cpp"), "-o", out, "-L" + os.path.join(root, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.check_call(cmd)
    spec = importlib.util.spec_from_file_location("_binding", out)
    module = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(module)
    lib = ctypes.PyDLL(out)

    def call(name, args, want):
        """Sizes the entry point saw in a call during which every argument tensor is reshaped."""
        def reshape():
            for t in args:
                if isinstance(t, torch.Tensor):
                    t.resize_(1, 1, 1, 1, 1, 1, t.numel())      # more dimensions than a tensor keeps inline
        ctypes.py_object.in_dll(lib, "callback").value = reshape
        assert getattr(module, name)(*args) == 0
        return list((ctypes.c_int * 8).in_dll(lib, "seen"))[:len(want)]

    return call


def bf16(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16)


def f32(*shape):
    return torch.zeros(shape)


@pytest.mark.parametrize("name", ["decode", "decode_multi", "gate", "prefill", "prefill_overlap"])
def test_sizes_are_those_at_the_time_of_the_call(recorder, name):
    if name == "decode":
        args = (bf16(3, 2, 128), bf16(3, 2, 128), bf16(3, 4, 128), f32(3, 4), f32(3, 4), f32(5, 4, 1, 1), None,
                bf16(3, 4, 128), 1.0, None)
        want = [3, 2, 4, 128, 128, 5]
    elif name == "decode_multi":
        args = (bf16(3, 7, 2, 128), bf16(3, 7, 2, 128), bf16(3, 7, 4, 128), f32(3, 7, 4), f32(3, 7, 4), f32(5, 4, 1, 1), None,
                bf16(3, 7, 4, 128), 1.0, 0, None)
        want = [3, 7, 2, 4, 128, 128, 5]
    elif name == "gate":
        args = (bf16(9, 4), bf16(9, 4), f32(4), f32(4), f32(9, 4), f32(9, 4))
        want = [9, 4]
    else:
        args = (5 if name == "prefill_overlap" else 0, bf16(9, 2, 128), bf16(9, 2, 128), bf16(9, 4, 128), f32(9, 4), f32(9, 4),
                torch.zeros(3, dtype=torch.int32), None, f32(2, 4, 1, 1), None, bf16(9, 4, 128), 1.0,
                torch.zeros(64, dtype=torch.uint8), 0, 64, None, -1)
        want, name = [9, 2, 2, 4, 128, 128, 2], "prefill"
    assert recorder(name, args, want) == want
