"""csrc/binding.cpp on a machine without a GPU: compiled with a stand-in for
torch's CUDA stream and a function that shows a host tensor as a CUDA one, so
that it takes ordinary arguments and calls whatever library it is handed.

Run as a program (path of the module): arguments whose memory cannot be
accessed, in every place of every function.
"""
import ctypes
import importlib.machinery
import importlib.util
import os
import subprocess
import sys
import sysconfig

import torch

import paper_2608_27370_gb300 as P

STREAM = 0x5EED
STUB = """#pragma once
namespace c10::cuda {
struct CUDAStream { void *stream() const { return reinterpret_cast<void *>(%d); } };
inline CUDAStream getCurrentCUDAStream() { return {}; }
}  // namespace c10::cuda
""" % STREAM
SOURCE = """#include "%s"
#include <ATen/ops/from_blob.h>
static PyObject *as_cuda(PyObject *, PyObject *o) {
    at::Tensor t = THPVariable_Unpack(o);
    const at::Device d(at::kCUDA, 0);
    return THPVariable_Wrap(at::from_blob(t.data_ptr(), t.sizes(), t.strides(), [t](void *) {}, t.options().device(d), d));
}
static PyMethodDef extra[] = {{"as_cuda", as_cuda, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyMODINIT_FUNC PyInit__harness() {
    PyObject *m = PyInit__native();
    if (m) PyModule_AddFunctions(m, extra);
    return m;
}
""" % P._build.BINDING


def build(folder) -> str:
    folder = str(folder)
    os.makedirs(os.path.join(folder, "c10", "cuda"))
    for name, text in (("c10/cuda/CUDAStream.h", STUB), ("harness.cpp", SOURCE)):
        with open(os.path.join(folder, name), "w") as f:
            f.write(text)
    torch_dir = os.path.dirname(torch.__file__)
    so = os.path.join(folder, "_harness.so")
    subprocess.run(["g++", "-O0", "-std=c++17", "-fPIC", "-shared", "-I", folder, '-DPURO_NATIVE_FOR="harness"',
                    "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
                    "-isystem", os.path.join(torch_dir, "include"), "-isystem",
                    os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
                    "-isystem", sysconfig.get_paths()["include"],
                    "-isystem", os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(P._build._nvcc()))), "include"),
                    "-I", P._build.INCLUDE, os.path.join(folder, "harness.cpp"), "-o", so,
                    "-L", os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"], check=True)
    return so


def load(so: str, library: dict):
    """The module, calling the functions at the addresses of `library` (name -> address)."""
    loader = importlib.machinery.ExtensionFileLoader("_harness", so)
    module = importlib.util.module_from_spec(importlib.util.spec_from_loader("_harness", loader))
    loader.exec_module(module)
    module.set_operand_type(P.FP8Operand)
    module.set_library(library)
    return module


class Recorder:
    """A library that notes its calls (name, arguments; operand structures by their fields)."""
    STATUS = 5
    OPERANDS = {"puro_fp8_linear_backward": (0, 1, 3, 4)}

    def __init__(self):
        self.calls, self.addresses, self.keep = [], {}, []
        for name, (res, types) in P._SIGNATURES.items():
            if res is not ctypes.c_int32:
                continue
            proto = ctypes.CFUNCTYPE(res, *types)
            where = self.OPERANDS.get(name, (0, 1) if name.startswith("puro_fp8_linear_") else ())
            note = proto(lambda *a, name=name, where=where: self._note(name, where, a))
            self.keep.append(note)
            self.addresses[name] = ctypes.cast(note, ctypes.c_void_p).value
            setattr(self, name, proto(self.addresses[name]))  # as a loaded library has it

    def _note(self, name, where, args):
        fields = [f for f, _ in P.puro_fp8_tensor_t._fields_]
        args = [[getattr(P.puro_fp8_tensor_t.from_address(a), f) for f in fields] if i in where and a else a
                for i, a in enumerate(args)]
        self.calls.append((name, args))
        return self.STATUS


def shown_as_cuda(module, arg):
    if torch.is_tensor(arg):
        return module.as_cuda(arg)
    if isinstance(arg, P.FP8Operand):
        return P.FP8Operand(module.as_cuda(arg.data), module.as_cuda(arg.scale), arg.fmt, arg.scaling, arg.role)
    return arg


def _check_unreadable_tensors(so: str) -> None:
    from test_binding import _buffers, _native_args

    def called(*_):
        print("called", flush=True)
        os._exit(1)

    called = ctypes.CFUNCTYPE(ctypes.c_int32)(called)
    module = load(so, {n: ctypes.cast(called, ctypes.c_void_p).value for n in P._SIGNATURES})
    for name, args in _native_args(_buffers("cpu")).items():
        fn, args = getattr(module, name), [shown_as_cuda(module, a) for a in args]
        for k, a in enumerate(args):
            for t in [a] if torch.is_tensor(a) else [a.data, a.scale] if isinstance(a, P.FP8Operand) else []:
                odd = module.as_cuda(torch.zeros(t.shape, dtype=t.dtype).as_strided(t.shape, t.stride())
                                     if t.is_contiguous() else
                                     torch.zeros((t.shape[0], t.stride(0)), dtype=t.dtype)[:, :t.shape[1]])
                torch._C._set_throw_on_mutable_data_ptr(odd)
                new = odd if t is a else P.FP8Operand(odd, a.scale) if t is a.data else P.FP8Operand(a.data, odd)
                assert fn(*args[:k], new, *args[k + 1:]) is None, (name, k)
                assert len([None] * 1000) == 1000  # (the interpreter still holds its lock)
    print("declined all", flush=True)


if __name__ == "__main__":
    _check_unreadable_tensors(sys.argv[1])
