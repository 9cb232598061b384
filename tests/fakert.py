"""Runs a piece of Python against the library's host side on the stand-in runtime of
tests/fake_cudart.c, in a child process (no GPU is used, on a GPU machine neither)."""
import ctypes as C
import os
import shutil
import subprocess
import sys
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


def run(code):
    """The child's standard output; raises with its error output if it fails."""
    with tempfile.TemporaryDirectory() as d:
        so = os.path.join(d, "fake_cudart.so")
        subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I", _include(), "-o", so,
                        os.path.join(HERE, "fake_cudart.c")], check=True, capture_output=True, text=True)
        from paper_1308_5992_gb300 import _build
        _build.build()
        env = dict(os.environ, LD_PRELOAD=so, FAKE_CUDART=so, PYTHONPATH=ROOT + os.pathsep + HERE)
        r = subprocess.run([sys.executable, "-c", "from fakert import *\n" + code], env=env, cwd=d, timeout=300,
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout


# ---------------------------------------------------------------- in the child
def fake():
    L = C.CDLL(os.environ["FAKE_CUDART"])
    for f in ("fake_dead_what", "fake_captured", "fake_launched"):
        getattr(L, f).restype = C.c_char_p
    L.fake_fail.argtypes = [C.c_size_t, C.c_size_t, C.c_int, C.c_int]
    L.fake_times.argtypes = [C.c_float, C.c_float]
    return L


class Hier:
    """A hierarchy of zeros on the lattices Nl, loaded from a file; vectors are one host buffer."""

    def __init__(self, Nl, **params):
        import numpy as np
        from oracle import hierfile
        from paper_1308_5992_gb300 import wilson_amg as W
        self.W, self.Nl = W, Nl
        self.lib = W.lib()
        hierfile.fnv1a64 = lambda data: self.lib.wl_hash_bytes(data, len(data))  # the same sum, compiled
        U = np.ones((2, Nl[0], Nl[0]), np.complex128)
        path = os.path.join(os.getcwd(), "h%s.wlh" % "_".join(map(str, Nl)))
        if not os.path.exists(path):
            hierfile.write(path, U, 0.1, Nl, [a // b for a, b in zip(Nl, Nl[1:])],
                  [np.zeros((n * n // 2, 2, 4)) for n in Nl[:-1]], [np.zeros((n * n // 2, 9, 2, 2)) for n in Nl[1:]])
        self.op, self.amg = C.c_void_p(), C.c_void_p()
        self.ok(self.lib.wilson_create(C.c_void_p(U.ctypes.data), Nl[0], 0.1, None, C.byref(self.op)))
        self.prm = W.amg_params_default(zero_guess=1, levels=len(Nl), block=[a // b for a, b in zip(Nl, Nl[1:])],
                                        **params)
        self.ok(self.lib.amg_import(self.op, path.encode(), C.byref(self.prm), C.byref(self.amg)))
        self.buf = np.zeros(64 * 2 * Nl[0] * Nl[0], np.complex128)

    def setup(self):
        """amg_setup on the same operator (its hierarchy is given back at once)"""
        out = C.c_void_p()
        rc = self.lib.amg_setup(self.op, C.byref(self.prm), C.byref(out))
        if rc == 0:
            self.lib.amg_destroy(out)
        return rc

    def close(self):
        self.lib.amg_destroy(self.amg)
        self.lib.wl_destroy(self.op)

    def ok(self, rc):
        assert rc == 0, (rc, self.lib.wl_last_error())

    @property
    def v(self):
        return C.c_void_p(self.buf.ctypes.data)

    def cycle(self, nrhs, prec):
        return self.lib.amg_cycle(self.amg, self.v, self.v, nrhs, prec)

    def solve(self, nrhs):
        return self.lib.amg_solve(self.amg, self.v, self.v, nrhs, 1e-12, None)

    def serve(self, slots):
        srv, cfg = C.c_void_p(), C.c_int()
        self.ok(self.lib.srv_create(1 << 36, slots, C.byref(srv)))
        self.ok(self.lib.srv_add(srv, self.amg, C.byref(cfg)))
        rc = self.lib.srv_start(srv)
        self.lib.srv_destroy(srv)
        return rc
