"""The library's own objects linked against a stand-in for the CUDA runtime
(fake_cudart/fake_cudart.c), for host tests of its launch logic: which kernels
a call launches, and what it does when a launch fails."""
import ctypes
import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
LAUNCH = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_char_p, ctypes.POINTER(ctypes.c_void_p))
MEMSET = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t)


def load(tmp_dir):
    """The library over the stand-in runtime, with the binding's signatures."""
    from paper_2405_01420_gb300 import build, nb
    build.build()
    objs = sorted(os.path.join(build.BUILD_DIR, os.path.basename(s)[:-3] + ".o")
                  for s in glob.glob(os.path.join(build.CSRC, "*.cu")))
    if not all(map(os.path.exists, objs)):  # a library that came without its objects
        build.build(force=True)
    out = os.path.join(str(tmp_dir), "libnb_fake.so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", out, *objs, "-x", "c", "-fPIC",
                    os.path.join(HERE, "fake_cudart", "fake_cudart.c"), "-lpthread"], check=True)
    lib = ctypes.CDLL(out)
    for name, (res, args) in nb.SIGNATURES.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    return lib


class Recorder:
    """Hooks that record the launches by kernel name. ``emulate(name, args)`` may act for a kernel;
    ``fail(name)`` and ``fail_memset()`` return a cudaError_t, 0 for success."""

    def __init__(self, lib, emulate=None):
        self.names, self.memsets = [], []
        self.emulate = emulate
        self.fail = lambda name: 0
        self.fail_memset = lambda: 0
        self._hooks = (LAUNCH(self._launch), MEMSET(self._memset))
        lib.fake_hooks(*self._hooks)

    def _launch(self, name, args):
        name = name.decode()
        self.names.append(name)
        e = self.fail(name)
        if e == 0 and self.emulate:
            self.emulate(name, args)
        return e

    def _memset(self, p, value, n):
        self.memsets.append((p, value, n))
        return self.fail_memset()
