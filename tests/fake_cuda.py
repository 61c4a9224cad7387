"""The library's host code on a CUDA runtime made for tests (tests/native): memory is host memory, kernels are recorded and
not run, failures are switched on.  Every FakeLibrary is a copy of its own, with its own kept memory."""
import ctypes as C
import functools
import os
import shutil
import subprocess
import tempfile

from paper_2607_20125_b200 import binding

NATIVE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
RELAXED, GLOBAL_MODE = 1, 2  # capture modes


@functools.lru_cache(maxsize=None)
def _built():
    folder = tempfile.TemporaryDirectory()
    lib = os.path.join(folder.name, "fake.so")
    cmd = [os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-cudart", "none", "-shared", "-Xcompiler", "-fPIC,-fno-gnu-unique", "-Xlinker", "-Bsymbolic",
           "-gencode", "arch=compute_100a,code=sm_100a", "-Xptxas", "-O0", "-std=c++17", "-o", lib,
           os.path.join(NATIVE, "headcast_on_fake_cuda.cu"), os.path.join(NATIVE, "fake_cuda.cpp")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stdout + res.stderr
    return folder, lib


class FakeLibrary:
    def __init__(self):
        folder, lib = _built()
        handle, path = tempfile.mkstemp(suffix=".so", dir=folder.name)
        os.close(handle)
        shutil.copy(lib, path)
        self.lib = binding.load_library(path)
        for name in ("fake_used", "fake_pool_unused", "fake_busy", "fake_busy_writes", "fake_stray_writes"):
            getattr(self.lib, name).restype = C.c_longlong
        self.lib.fake_capacity_left.argtypes = [C.c_longlong]
        self.lib.fake_capture.argtypes = [C.c_int, C.c_void_p]
        self.lib.fake_is_live.argtypes = [C.c_void_p]
        self.lib.fake_attn_part_o.restype = C.c_void_p
        self.lib.fake_log.restype = C.c_char_p
        self.lib.fake_reset()

    def __getattr__(self, name):  # used(), capture(mode, stream), ...
        return getattr(self.lib, "fake_" + name)

    def context(self, **cfg):
        return FakeContext(self.lib, **cfg)


class FakeContext:
    """One context; tensors are an address that nothing reads.  Methods return the status code."""

    def __init__(self, lib, **cfg):
        self.lib = lib
        self.cfg = binding.default_config(**cfg)
        self.ptr = C.c_void_p()
        self.rc = lib.headcast_create(C.byref(self.cfg), C.byref(self.ptr))
        self.buffer = C.create_string_buffer(64)
        self.tensor = (C.addressof(self.buffer) + 15) & ~15

    def append(self, blocks=1, stream=0):
        for _ in range(blocks):
            rc = self.lib.headcast_append(self.ptr, self.tensor, self.tensor, stream)
            if rc:
                return rc
        return 0

    def split(self, labels, stream=0):
        rc = self.lib.headcast_set_labels(self.ptr, (C.c_int32 * len(labels))(*labels))
        return rc or self.lib.headcast_split_cache(self.ptr, stream)

    def full_attend(self, stream=0):
        return self.lib.headcast_full_attend(self.ptr, self.tensor, self.tensor, stream)

    def attend(self, stream=0):
        return self.lib.headcast_attend(self.ptr, self.tensor, self.tensor, stream)

    def attend_host(self, stream=0):
        return self.lib.headcast_attend_host(self.ptr, self.tensor, self.tensor, stream)

    def classify(self, stream=0):
        return self.lib.headcast_classify(self.ptr, self.tensor, (C.c_int32 * self.cfg.n_heads)(), None, stream)

    def export(self, head=0, stream=0):
        return self.lib.headcast_export_cache(self.ptr, head, self.tensor, self.tensor, None, stream)

    def destroy(self):
        rc = self.lib.headcast_destroy(self.ptr)
        self.ptr = C.c_void_p()
        return rc
