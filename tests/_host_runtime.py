"""The library's host code on a CUDA runtime without a device (host_runtime/
fake_cuda.cpp): kernels do nothing, every call that touches a stream, memory or an
event is logged.  For tests of what the host enqueues, in which order, on CPU."""
import contextlib
import ctypes
import glob
import json
import os
import subprocess

import numpy as np

import paper_2007_06048_gb300 as M
from paper_2007_06048_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = [os.path.join(HERE, "host_runtime", f) for f in ("fake_cuda.cpp", "step_arguments.cu")]
OUT = os.path.join(_build.ROOT, "_build", "host_runtime")
LIB = os.path.join(OUT, "libmmod_host_runtime.so")


def _objects():
    return [os.path.join(_build.OBJDIR, os.path.basename(s)[:-3] + ".o") for s in _build._sources()]


def build():
    M.build()
    if not all(os.path.exists(o) for o in _objects()):
        _build.build(force=True)
    newest = max(os.path.getmtime(p) for p in [*SRC, *_objects()])
    if os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    os.makedirs(OUT, exist_ok=True)
    objs = [os.path.join(OUT, os.path.basename(src) + ".o") for src in SRC]
    for src, obj in zip(SRC, objs):
        subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-c", src, "-o", obj], check=True)
    tmp = LIB + f".tmp{os.getpid()}"
    # -Bsymbolic: the functions here, not those of a CUDA runtime in the process
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic,-z,defs", "-o", tmp, *_objects(), *objs], check=True)
    os.replace(tmp, LIB)
    return LIB


class Runtime:
    def __init__(self, lib):
        self.lib = lib
        lib.fake_log.restype = ctypes.c_char_p
        lib.fake_malloc.restype = lib.fake_stream.restype = ctypes.c_void_p
        lib.fake_malloc.argtypes = lib.fake_fail_malloc.argtypes = [ctypes.c_size_t]
        lib.fake_free.argtypes = [ctypes.c_void_p]
        lib.fake_fast_kernel.argtypes = [ctypes.c_char_p]
        self.open = []
        self.reset()

    def propagator(self, p, model=True):
        """A propagator of problem p, closed when the runtime is left."""
        prop = M.Propagator.from_problem(p)
        self.open.append(prop)
        if model:
            prop.set_model(np.ascontiguousarray(p.vel))
        return prop

    def batch(self, props):
        b = M.Batch(props)
        self.open.append(b)
        return b

    def close(self):
        while self.open:
            self.open.pop().close()

    def reset(self):
        self.lib.fake_fail_encode(0, 0, 0)
        self.lib.fake_fail_malloc(0)
        self.lib.fake_fast_kernel(b"")
        self.lib.fake_clear()

    def malloc(self, floats):
        return self.lib.fake_malloc(4 * max(int(floats), 1))

    def free(self, ptr):
        self.lib.fake_free(ptr)

    def stream(self):
        return self.lib.fake_stream()

    def log(self, clear=True):
        """The calls since the last clear, as dicts."""
        out = [json.loads(line) for line in self.lib.fake_log().decode().splitlines()]
        if clear:
            self.lib.fake_clear()
        return out


@contextlib.contextmanager
def host_runtime():
    """The package on the runtime without a device."""
    path = build()
    real, real_path = M._lib, _build.LIB
    try:
        M._lib, _build.LIB = None, path
        rt = Runtime(M.load())
        try:
            yield rt
        finally:
            rt.close()   # handles of this runtime never reach the real library
            rt.reset()
    finally:
        M._lib, _build.LIB = real, real_path
