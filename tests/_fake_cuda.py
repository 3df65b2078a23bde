"""The library linked with a stand-in for the CUDA runtime (fake_cuda.cpp): its host paths without a GPU."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST, DEVICE, MANAGED = 1, 2, 3            # cudaMemoryType


class Fake:
    """The library (attribute L) and what it asked of the runtime."""

    def __init__(self, path):
        self.L = ctypes.CDLL(path, mode=os.RTLD_LOCAL | os.RTLD_NOW)
        self.L.fake_log.restype = ctypes.c_char_p
        self.L.fake_live.restype = ctypes.c_size_t
        self.L.fake_memory.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_int]
        self._hook = None

    def reset(self):
        self.L.fake_clear()
        self.L.fake_fail(b"", 0, 0)
        self.L.fake_device(0)
        self.hook(None)

    def calls(self, name=None):
        """The calls so far, split into words; those of one name only if one is given."""
        lines = [c.split() for c in self.L.fake_log().decode().splitlines()]
        return [c for c in lines if name is None or c[0] == name]

    def launches(self, kernel):
        return [c for c in self.calls("launch") if kernel in c[1]]

    def clear(self):
        self.L.fake_clear()

    def fail(self, name, nth=1, err=2):
        """The nth call of `name` from here on returns err (2: out of memory)."""
        self.L.fake_fail(name.encode(), nth if name else 0, err)

    def memory(self, address, nbytes, kind=DEVICE, device=0):
        """An address that the runtime knows and nothing touches; nbytes 0 forgets it."""
        self.L.fake_memory(address, nbytes, kind, device)

    def hook(self, f):
        """f(kernel name, pointers to the arguments) at every launch."""
        proto = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.POINTER(ctypes.c_void_p))
        self._hook = proto(f) if f else proto()
        self.L.fake_hook(self._hook)


def build(out_dir):
    from paper_2209_14889_gb300 import _build
    objs = [os.path.join(_build.BUILD, s.replace(".cu", ".o")) for s in _build.SOURCES]
    _build.build(force=not all(os.path.exists(o) for o in objs))
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    lib = os.path.join(str(out_dir), "libvlb_fake.so")
    # -Bsymbolic: torch brings a runtime of its own into the process
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", inc, "-o", lib,
                    os.path.join(ROOT, "tests", "fake_cuda.cpp"), *objs], check=True, capture_output=True)
    return Fake(lib)
