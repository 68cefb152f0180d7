"""The library's host code (lbm_api.cu, lbm_batch.cu) linked against a fake CUDA runtime and fake step-kernel
launches: which launches a call makes, and what it does when one of them fails, without a GPU."""
import ctypes as C
import os
import subprocess

from paper_2408_15654_gb300 import build as _build
from paper_2408_15654_gb300 import lbm

HERE = os.path.dirname(os.path.abspath(__file__))
FIELDS = ("kind", "status", "nsteps", "cooperative", "ctas", "members", "steps", "tiles")
SMS = 152


def build(out_dir: str):
    """Compile and link; the library with the prototypes of the real one where it has the entry points."""
    _build.build()
    objs = [os.path.join(_build.BUILD_DIR, f"{n}.cu.o") for n in ("lbm_api", "lbm_batch")]
    if not all(os.path.exists(o) and os.path.getmtime(o) >= max(map(os.path.getmtime, _build._deps())) for o in objs):
        objs = []
        for n in ("lbm_api", "lbm_batch"):
            objs.append(os.path.join(out_dir, n + ".o"))
            subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-c", os.path.join(_build.CSRC, n + ".cu"),
                            "-o", objs[-1]], check=True)
    launch, runtime, path = (os.path.join(out_dir, n) for n in ("launch.o", "runtime.o", "libfake.so"))
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-c", os.path.join(HERE, "fake_launch.cu"), "-o",
                    launch], check=True)
    subprocess.run(["g++", "-O1", "-fPIC", "-c", os.path.join(HERE, "fake_runtime.cpp"), "-o", runtime], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", path, *objs, launch, runtime, "-lpthread"],
                   check=True)
    lib = C.CDLL(path)
    lib.lbm_last_error.restype = C.c_char_p
    return lib


class Fake:
    """One linked library; ``lattice`` and ``batch`` make handles on addresses that nobody reads."""

    def __init__(self, out_dir):
        self.lib = build(out_dir)
        self._handles = []

    def ok(self, rc):
        assert rc == lbm.LBM_OK, self.lib.lbm_last_error()

    def reset(self):
        self.lib.fake_reset()

    def fail(self, kind, at, code):
        """The ``at``-th launch of this kind from now on returns ``code``."""
        self.lib.fake_fail(ord(kind), at, code)

    def prepared(self, kind):
        return self.lib.fake_prepared(ord(kind))

    def launches(self):
        out, v = [], (C.c_longlong * len(FIELDS))()
        for k in range(self.lib.fake_count()):
            self.lib.fake_get(k, v)
            out.append(dict(zip(FIELDS, v), kind=chr(v[0])))
        return out

    def lattice(self, p, init=True):
        q, n, h = lbm.make_params(p), C.c_size_t(), C.c_void_p()
        self.ok(self.lib.lbm_workspace_bytes(C.byref(q), C.byref(n)))
        self.ok(self.lib.lbm_create(C.byref(q), C.c_void_p(1 << 32), n, C.c_void_p(64), C.byref(h)))
        if init:
            f = C.c_void_p(1 << 33)
            self.ok(self.lib.lbm_init_fields(h, f, f, f, f, f, lbm.LBM_MEM_DEVICE))
        return h

    def step(self, h, n):
        return self.lib.lbm_step(h, C.c_int64(n))

    def steps(self, h):
        v = C.c_int64()
        self.ok(self.lib.lbm_steps_taken(h, C.byref(v)))
        return v.value

    def batch(self, members, capacity=None):
        arr, n, b, t = (C.c_void_p * len(members))(*members), C.c_size_t(), C.c_void_p(), C.c_int64()
        capacity = capacity or len(members)
        self.ok(self.lib.lbm_batch_tiles(arr, len(members), C.byref(t)))
        self.ok(self.lib.lbm_batch_workspace_bytes(capacity, t, C.byref(n)))
        self.ok(self.lib.lbm_batch_create(capacity, t, C.c_void_p(1 << 34), n, C.c_void_p(64), C.byref(b)))
        self.ok(self.lib.lbm_batch_set_members(b, arr, len(members)))
        return b

    def batch_step(self, b, n):
        return self.lib.lbm_batch_step(b, C.c_int64(n))
