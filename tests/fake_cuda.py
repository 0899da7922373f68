"""Runs a test of the library's host code in a child process whose CUDA runtime
is tests/native/fake_cudart.cpp (host memory, two devices, no kernels)."""
import os
import subprocess
import sys
import tempfile
import textwrap

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes as C
fake = C.CDLL({fake!r}, mode=C.RTLD_GLOBAL)
lib = C.CDLL({lib!r})
fake.fake_capacity.argtypes = [C.c_size_t]
fake.fake_used.restype = fake.fake_idle.restype = C.c_size_t
for f in ("fake_max_persistent_grid",):
    getattr(fake, f).restype = C.c_uint
lib.vd_last_error.restype = C.c_char_p
P = C.c_void_p
F = C.c_float


def dev(n):
    p = P()
    assert fake.cudaMalloc(C.byref(p), C.c_size_t(n)) == 0
    return p


def ok(status):
    assert status == 0, (status, lib.vd_last_error())
"""

_built = {}


def run(body):
    """Runs `body` (with the prelude's names) and returns its standard output."""
    from paper_2104_06800_gb300 import build
    if not _built:
        cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc_path())), "include")
        out = os.path.join(tempfile.mkdtemp(), "libfake_cudart.so")
        subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", cuda,
                        os.path.join(ROOT, "tests", "native", "fake_cudart.cpp"), "-o", out],
                       check=True)
        _built["fake"] = out
        _built["lib"] = build.build()
    code = PRELUDE.format(**_built) + textwrap.dedent(body)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-3000:]
    return r.stdout
