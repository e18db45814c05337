"""The library on a CUDA runtime without a GPU (fake_cudart.c): its calls and
launches in order, and how much memory each pointer that it hands to a kernel
really has.  For processes of their own (host_call): the real runtime must not
be loaded beside it."""
import ctypes as C
import json
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
STREAM = 0x5EA0          # a stream of the program's own
REPORT = C.CFUNCTYPE(None, C.c_char_p, C.c_void_p, C.c_void_p, C.c_size_t, C.POINTER(C.c_uint), C.POINTER(C.c_void_p))


class Fake:
    def __init__(self, workdir):
        so = os.path.join(workdir, "libcudart.so.13")
        ver = os.path.join(workdir, "version.map")
        with open(ver, "w") as f:
            f.write("libcudart.so.13 { global: *; };\n")
        subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-Wall", "-Werror", "-Wl,-soname,libcudart.so.13",
                        f"-Wl,--version-script={ver}", "-o", so, os.path.join(HERE, "fake_cudart.c")], check=True)
        self.rt = C.CDLL(so, mode=C.RTLD_GLOBAL)
        self.rt.fake_room.argtypes, self.rt.fake_room.restype = [C.c_void_p], C.c_size_t
        self.calls = []          # (name, stream, bytes, grid)
        self.on_launch = None    # called with (name, grid, args) while a launch's arguments are alive
        self._cb = REPORT(self._report)
        self.rt.fake_report(self._cb)
        sys.path.insert(0, os.path.dirname(HERE))

    def _report(self, name, stream, ptr, nbytes, grid, args):
        g = tuple(grid[i] for i in range(3)) if grid else None
        self.calls.append((name.decode(), stream or 0, nbytes, g))
        if g and self.on_launch:
            self.on_launch(name.decode(), g, args)

    def clear(self):
        self.calls = []

    def room(self, p):
        """Bytes of device memory from p on (0: not device memory)."""
        return self.rt.fake_room(p)

    def device(self, nbytes):
        p = C.c_void_p()
        assert self.rt.cudaMalloc(C.byref(p), C.c_size_t(nbytes)) == 0
        return p.value

    def names(self):
        return [c[0] for c in self.calls]

    def launches(self):
        return [c for c in self.calls if c[3]]


def host_call(script, what, workdir, timeout=300):
    """`python script what` in a process of its own; the JSON it prints last."""
    r = subprocess.run([sys.executable, script, what, str(workdir)], capture_output=True, text=True, timeout=timeout)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.splitlines()[-1])
